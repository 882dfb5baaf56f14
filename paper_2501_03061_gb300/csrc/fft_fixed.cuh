// Compile-time-size FFTs on 2-D tiles in shared memory, for cubic grids whose side N is known at compile
// time.
//
// A line of N = N1 N2 points (the split and index maps of fft_reg.cuh) is transformed in two stages of short
// transforms held in registers: N1 points in place for every n2, then N2 points for every k1, written in
// natural order. Coprime splits have no twiddles between the stages. Threads are laid out with the line index
// fastest, so both tile orientations are free of bank conflicts. Against radix stages of 8, 4, 5, 3 and 2 this
// takes two passes over shared memory instead of two to four, three barriers instead of four to eight, and a fifth to
// two fifths fewer operations (24 = 3 x 8: 13 per point and axis against 19, 48 = 3 x 16: 16 against 27), which is
// what bounds the FP64 forms.
#pragma once

#include "fft.cuh"
#include "fft_reg.cuh"

namespace pt {

// odd row pitch (in elements) of an N x N tile
template <int N>
constexpr int kPitch = (N % 2 == 0) ? N + 1 : N;

// transform of NLINES lines of N points; element (line, pos) at buf[line*LS + pos*PS], tw[k] = exp(-2 pi i k / N)
template <int N, bool INV, int NT, int NLINES, int LS, int PS, class T>
__device__ __forceinline__ void cfft_lines(cx<T>* buf, const cx<T>* tw) {
  using L = rl::Line<N>;
  constexpr int N1 = L::N1, N2 = L::N2;
  constexpr bool pfa = L::P::pfa;
  const int tid = threadIdx.x;
  auto wrap = [](int i) { return i < N ? i : i - N; };
  constexpr int TOTAL1 = N2 * NLINES;
#pragma unroll 1
  for (int f = tid; f < TOTAL1; f += NT) {
    const int line = f % NLINES, n2 = f / NLINES;
    cx<T>* p = buf + line * LS;
    auto at = [&](int n1) -> cx<T>& { return p[(pfa ? wrap(N1 * n2 + N2 * n1) : n1 * N2 + n2) * PS]; };
    cx<T> v[N1];
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) v[n1] = at(n1);
    rl::short_dft<N1, INV>(v);
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
      if (!pfa && k1 > 0) {
        cx<T> w = tw[k1 * n2];
        if (INV) w.im = -w.im;
        v[k1] = cmul(v[k1], w);
      }
      at(k1) = v[k1];
    }
  }
  __syncthreads();
  constexpr int TOTAL2 = N1 * NLINES, BPT = (TOTAL2 + NT - 1) / NT;
  cx<T> v[BPT][N2];
#pragma unroll
  for (int u = 0; u < BPT; ++u) {
    const int f = tid + u * NT;
    if (TOTAL2 % NT == 0 || f < TOTAL2) {
      const int line = f % NLINES, k1 = f / NLINES;
      const cx<T>* p = buf + line * LS;
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) v[u][n2] = p[(pfa ? wrap(N2 * k1 + N1 * n2) : k1 * N2 + n2) * PS];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < BPT; ++u) {
    const int f = tid + u * NT;
    if (TOTAL2 % NT == 0 || f < TOTAL2) {
      const int line = f % NLINES, k1 = f / NLINES;
      cx<T>* p = buf + line * LS;
      rl::short_dft<N2, INV>(v[u]);
      const int b1 = pfa ? (L::P::freq(1, 0) * k1) % N : k1;
#pragma unroll
      for (int k2 = 0; k2 < N2; ++k2) p[(pfa ? wrap(b1 + L::P::freq(0, k2)) : b1 + N1 * k2) * PS] = v[u][k2];
    }
  }
  __syncthreads();
}

// transforms of an N x N tile with rows of pitch kPitch<N>: along the fast axis (within rows)
// and along the slow axis (within columns)
template <int N, bool INV, int NT, class T>
__device__ __forceinline__ void cfft_fast(cx<T>* buf, const cx<T>* tw) {
  cfft_lines<N, INV, NT, N, kPitch<N>, 1>(buf, tw);
}
template <int N, bool INV, int NT, class T>
__device__ __forceinline__ void cfft_slow(cx<T>* buf, const cx<T>* tw) {
  cfft_lines<N, INV, NT, N, 1, kPitch<N>>(buf, tw);
}

// sides with compile-time kernels (cubic grids); others use the runtime-plan kernels
#define PT_FIXED_SIZES(X) X(16) X(20) X(24) X(30) X(32) X(36) X(40) X(48) X(54) X(60) X(64)

inline bool fixed_cubic(const pt_grid& g) {
  if (g.nx != g.ny || g.nx != g.nz) return false;
  switch (g.nx) {
#define PT_CASE(n) case n:
    PT_FIXED_SIZES(PT_CASE)
#undef PT_CASE
    return true;
    default:
      return false;
  }
}

}  // namespace pt
