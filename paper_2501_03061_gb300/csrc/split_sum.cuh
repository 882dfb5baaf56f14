// Sum of the split partials of a Gram entry: the CTA's 256 threads are E = 256 / G consecutive entries times
// G groups of splits.  A single thread per entry read its splits one after another: 48 x 48 entries in 152
// splits took 72 us on nine CTAs.
#pragma once

#include "common.cuh"

namespace pt {

constexpr int SUM_THREADS = 256;

// groups per entry: about ten partials to a thread
inline int split_groups(int nsplit) { return nsplit >= 48 ? 16 : nsplit >= 12 ? 4 : 1; }

// the entry of this thread
template <int G>
__device__ __forceinline__ size_t split_entry() {
  return size_t(blockIdx.x) * (SUM_THREADS / G) + threadIdx.x % (SUM_THREADS / G);
}

// sum_s load(s) over 0 <= s < nsplit, complete (in a fixed order) in the threads for which it returns true; every
// thread of the CTA calls it
template <int G, class F>
__device__ __forceinline__ bool split_sum(int nsplit, bool valid, F&& load, double& re, double& im) {
  constexpr int E = SUM_THREADS / G;
  const int x = threadIdx.x % E, g = threadIdx.x / E;
  re = im = 0.0;
  if (valid) {
#pragma unroll 4
    for (int s = g; s < nsplit; s += G) {
      const c128 v = load(s);
      re += v.re;
      im += v.im;
    }
  }
  if constexpr (G > 1) {
    __shared__ c128 red[G][E];
    red[g][x] = c128{re, im};
    __syncthreads();
    if (g == 0) {
      for (int q = 1; q < G; ++q) {
        re += red[q][x].re;
        im += red[q][x].im;
      }
    }
  }
  return g == 0 && valid;
}

}  // namespace pt

// Launch KERNEL<G> over n entries with the groups that nsplit asks for
#define PT_LAUNCH_SPLIT_SUM(KERNEL, n, ny, nsplit, stream, ...)                                                        \
  do {                                                                                                                 \
    const int g_ = ::pt::split_groups(nsplit), e_ = ::pt::SUM_THREADS / g_;                                            \
    const dim3 grid_(unsigned((size_t(n) + e_ - 1) / e_), ny);                                                         \
    if (g_ == 16) PT_LAUNCH(KERNEL<16>, grid_, ::pt::SUM_THREADS, 0, stream, __VA_ARGS__);                             \
    else if (g_ == 4) PT_LAUNCH(KERNEL<4>, grid_, ::pt::SUM_THREADS, 0, stream, __VA_ARGS__);                          \
    else PT_LAUNCH(KERNEL<1>, grid_, ::pt::SUM_THREADS, 0, stream, __VA_ARGS__);                                       \
  } while (0)
