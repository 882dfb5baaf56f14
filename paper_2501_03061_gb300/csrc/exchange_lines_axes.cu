// FP32 pair-FFT exchange with whole lines in registers on grids that are not cubic (exchange_lines.cu has the
// method), for axes of the lengths of PT_LINE_SIZES.
#include "exchange_lines.cuh"

namespace pt {

namespace {

// ---- the plane pass of a grid that is not cubic, axis by axis ------------------------------------
//
// A plane of nx x ny points needs both lengths at compile time in one kernel; one kernel per axis and
// length needs 16 of each instead of 256 of both, for two more round trips of a pair field (0.015 ns per
// pair and point against the cubic form's 0.008).  36 x 50 x 48, N = 33: 0.73 ms against 7.53 ms of the
// general kernels (exchange.cu), which keep their radix plans in registers and transform a symmetric pair's
// planes back once per target; those remain for axes below 16 points and for FP64.

// y lines of a pair field in place: thread (x, z)
template <int N, bool INV>
__global__ void __launch_bounds__(ZT, zmin(N)) k_xl_y(Tile t, const double* __restrict__ occ, c64* __restrict__ scratch, int nx,
                                                      int nz) {
  const int a = blockIdx.z, b = blockIdx.y;
  if (t.diag && b < a) return;
  const int p = blockIdx.x * ZT + threadIdx.x;
  if (p >= nx * nz) return;
  const int z = p / nx, x = p - z * nx;
  c64* f = scratch + (size_t(a * t.nj + b) * nz + z) * (size_t(N) * nx) + x;
  c64 v[N];
  const bool live = pair_live(t, occ, a, b);
  sfor<N>([&](auto q) { v[q] = ld_early(f + (INV ? Line<N>::freq(q) : int(q)) * nx); });
  if (!live) return;
  if constexpr (INV) Line<N>::inverse(v);
  else Line<N>::forward(v);
  sfor<N>([&](auto q) { f[(INV ? int(q) : Line<N>::freq(q)) * nx] = v[q]; });
}

// x lines of a pair field, times K/Ng, and back: thread (ky, kz), the rows of a CTA staged in shared memory.
// kt: K/Ng as [kz][kx][ky]
constexpr int XR = 64;  // rows per CTA
template <int N>
constexpr int kXPitch = N | 1;  // odd: rows at 8 bytes on distinct banks
template <int N>
__global__ void __launch_bounds__(XR, N <= 32 ? 10 : N <= 40 ? 8 : 6) k_xl_x(Tile t, const double* __restrict__ occ, const float* __restrict__ kt,
                                             c64* __restrict__ scratch, int ny, int nz) {
  __shared__ c64 buf[XR * kXPitch<N>];
  const int a = blockIdx.z, b = blockIdx.y;
  if ((t.diag && b < a) || !pair_live(t, occ, a, b)) return;
  const int r0 = blockIdx.x * XR, rows = min(XR, ny * nz - r0);
  c64* f = scratch + (size_t(a * t.nj + b) * ny * nz + r0) * N;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int e = i * XR + threadIdx.x, r = e / N;
    if (r < rows) buf[e + r * (kXPitch<N> - N)] = f[e];
  }
  __syncthreads();
  if (int(threadIdx.x) < rows) {
    c64* row = buf + threadIdx.x * kXPitch<N>;
    const int r = r0 + threadIdx.x, z = r / ny, y = r - z * ny;
    const float* k = kt + size_t(z) * N * ny + y;
    c64 v[N];
    sfor<N>([&](auto n) { v[n] = row[n]; });
    Line<N>::forward(v);
    sfor<N>([&](auto q) {
      constexpr int kx = Line<N>::freq(q);
      v[q] = v[q] * k[(kx < N - kx ? kx : N - kx) * ny];
    });
    Line<N>::inverse(v);
    sfor<N>([&](auto n) { row[n] = v[n]; });
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int e = i * XR + threadIdx.x, r = e / N;
    if (r < rows) f[e] = buf[e + r * (kXPitch<N> - N)];
  }
}

template <int N>
void run_y(const Tile& t, const double* occ, c64* scratch, int nx, int nz, bool inv, cudaStream_t st) {
  const dim3 grid((nx * nz + ZT - 1) / ZT, t.nj, t.ni);
  if (inv) PT_LAUNCH((k_xl_y<N, true>), grid, ZT, 0, st, t, occ, scratch, nx, nz);
  else PT_LAUNCH((k_xl_y<N, false>), grid, ZT, 0, st, t, occ, scratch, nx, nz);
}

template <int N>
void run_x(const Tile& t, const double* occ, const float* kt, c64* scratch, int ny, int nz, cudaStream_t st) {
  PT_LAUNCH(k_xl_x<N>, dim3((ny * nz + XR - 1) / XR, t.nj, t.ni), XR, 0, st, t, occ, kt, scratch, ny, nz);
}

}  // namespace

bool line_length(int n) {
  switch (n) {
#define PT_CASE(s) case s:
    PT_LINE_SIZES(PT_CASE)
#undef PT_CASE
    return true;
    default:
      return false;
  }
}

#define PT_SWITCH(n, CALL)                                             \
  switch (n) {                                                         \
    PT_LINE_SIZES(CALL)                                                \
    default:                                                           \
      fail(PT_INVALID_ARG, "no line kernels for this axis length");    \
  }

void exchange_tile_axes(const pt_grid& g, const Tile& t, const c64* src, const c64* tgt, const double* occ, const float* kt,
                        c64* scratch, c64* out, int sms, cudaStream_t st) {
  const int C = g.nx * g.ny;
#define PT_CASE(n) case n: run_zfwd<n, 0>(t, src, tgt, occ, scratch, C, st); break;
  PT_SWITCH(g.nz, PT_CASE)
#undef PT_CASE
#define PT_CASE(n) case n: run_y<n>(t, occ, scratch, g.nx, g.nz, false, st); break;
  PT_SWITCH(g.ny, PT_CASE)
#undef PT_CASE
#define PT_CASE(n) case n: run_x<n>(t, occ, kt, scratch, g.ny, g.nz, st); break;
  PT_SWITCH(g.nx, PT_CASE)
#undef PT_CASE
#define PT_CASE(n) case n: run_y<n>(t, occ, scratch, g.nx, g.nz, true, st); break;
  PT_SWITCH(g.ny, PT_CASE)
#undef PT_CASE
#define PT_CASE(n) case n: run_accum<n, 0>(t, src, occ, scratch, out, C, sms, st); break;
  PT_SWITCH(g.nz, PT_CASE)
#undef PT_CASE
}

}  // namespace pt
