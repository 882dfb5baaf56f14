// FP32 pair-FFT exchange on cubic grids (the sides of PT_FIXED_SIZES) with whole lines in registers
// (Sec. IV-A1, Eq. vxdiag; Algorithm 2 with sigma diagonalised).
//
// Three passes per tile of pairs (i, j), on one scratch field per pair:
//   zfwd:   a thread holds one z line of conj(src_i) tgt_j and transforms it (no shared memory);
//   plane:  a thread holds one y line of a kz plane, then one x line, multiplies by K(G)/Ng and goes
//           back; the plane turns twice through shared memory;
//   accum:  a thread owns one z line of one target: it transforms back the line of every pair that
//           feeds the target and adds d_c partner_c v to the line's sum, which stays on the SM.
// Transforming z first leaves only z lines for the last pass, so the potential v_ij is never written:
// a pair field crosses memory four times (written and read between the passes), where the tile
// kernels of exchange_fixed_kernels.cuh write and read it eight times.  A symmetric pair's z lines are
// transformed back once for each of its two targets (one transform in six done twice), which costs
// less than the write and the two reads of v_ij that it saves.
//
// What bounds it: registers.  A 64-point line is 128 registers, so an SM holds 12 warps (N <= 32: 20),
// and the passes run at 30-45% of the issue rate and 45-75% of the L1 rate, waiting on the loads
// and stores of lines between the transforms.  Measured on GB300, one V_x application, all pairs
// symmetric (this form against the tile kernels, at 64 against the TMA pipeline it replaced):
//   24^3 N = 64   0.22 against 0.67 ms      48^3 N = 128   6.7 against 18.0 ms
//   36^3 N = 96   1.83 against 4.66 ms      64^3 N = 96   11.0 against 14.4 ms
// i.e. 0.007-0.009 ns per pair and grid point against 0.012 (64^3) and 0.020-0.026.
#include <algorithm>

#include "exchange_sched.h"
#include "fft_fixed.cuh"
#include "fft_reg.cuh"
#include "internal.h"

namespace pt {

namespace {

using rl::Line;
using rl::sfor;

constexpr int MAXB = 128;  // largest pair-tile side

// One tile of the pair schedule: sources i0 .. i0 + ni, targets j0 .. j0 + nj, the field of pair
// (i0 + a, j0 + b) in slot a nj + b.  In the symmetric case a diagonal tile (diag) holds the pairs
// a <= b, and the pairs of an off-diagonal tile feed both their orbitals.  first: the tile's
// targets have no earlier tile.
struct Tile {
  int i0, ni, j0, nj, sym, diag, first;
};

__device__ __forceinline__ bool is_zero(const double* d) { return (__double_as_longlong(*d) << 1) == 0; }

// whether pair (a, b) of the tile feeds any target (its occupations are not all exactly zero)
__device__ __forceinline__ bool pair_live(const Tile& t, const double* occ, int a, int b) {
  const int i = t.i0 + a, j = t.j0 + b;
  return !(is_zero(occ + i) && (!t.sym || is_zero(occ + j)));
}

// a load that stays where it is written: ahead of the test of the pair's occupations, so that the two
// memory latencies of a CTA's start run together
__device__ __forceinline__ c64 ld_early(const c64* p) {
  c64 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.re), "=f"(v.im) : "l"(p));
  return v;
}

// ---- zfwd ----------------------------------------------------------------------------------

constexpr int ZT = 128;  // threads per CTA
// CTAs per SM: what the registers of a line allow without spills
constexpr int zmin(int n) { return n <= 24 ? 6 : n <= 32 ? 5 : n <= 40 ? 4 : 3; }

// rho = conj(src_i) tgt_j on one column, forward z transform
template <int N>
__global__ void __launch_bounds__(ZT, zmin(N)) k_xl_zfwd(Tile t, const c64* __restrict__ src, const c64* __restrict__ tgt,
                                                         const double* __restrict__ occ, c64* __restrict__ scratch) {
  constexpr int C = N * N;
  constexpr size_t NG = size_t(N) * C;
  const int a = blockIdx.z, b = blockIdx.y;
  if (t.diag && b < a) return;
  const int p = blockIdx.x * ZT + threadIdx.x;
  if (C % ZT && p >= C) return;
  const c64* x = src + size_t(t.i0 + a) * NG + p;
  const c64* y = tgt + size_t(t.j0 + b) * NG + p;
  c64* f = scratch + size_t(a * t.nj + b) * NG + p;
  c64 v[N];
  const bool live = pair_live(t, occ, a, b);
  sfor<N>([&](auto n) { v[n] = cmulc(ld_early(x + n * C), ld_early(y + n * C)); });
  if (!live) return;
  Line<N>::forward(v);
  sfor<N>([&](auto q) { f[Line<N>::freq(q) * C] = v[q]; });
}

// ---- plane ---------------------------------------------------------------------------------

// planes per CTA: N threads a plane, as many planes as fill whole warps
constexpr int planes(int n) {
  return n == 20 ? 10 : n == 16 || n == 24 || n == 36 || n == 40 ? 4 : n == 30 || n == 32 || n == 48 ? 2 : 1;
}
// row pitch of a plane's transpose buffer: 2 mod 4, so that both the column accesses (8 bytes, lanes on
// consecutive columns) and the row accesses (16 bytes, lanes on consecutive rows) are free of conflicts
constexpr int plane_pitch(int n) { return n % 4 == 0 ? n + 2 : n; }
// bytes between the buffers of a CTA's planes: padded so that the column accesses of a warp that spans two
// planes run on over the banks
constexpr int plane_stride(int n) {
  const int words = 2 * n * plane_pitch(n);
  return 4 * (words + ((2 * n - words) % 32 + 32) % 32);
}
template <int N>
constexpr int kPlaneThreads = (planes(N) * N + 31) / 32 * 32;
template <int N>
constexpr size_t kPlaneSmem = size_t(planes(N)) * plane_stride(N);
template <int N>
constexpr int plane_min() {  // CTAs per SM by registers (a line and its transform without spills) and shared memory
  const int regs = N <= 24 ? 80 : N == 30 ? 104 : N <= 32 ? 96 : N <= 40 ? 128 : 168;
  const int by_regs = 65536 / (regs * kPlaneThreads<N>);
  const int by_smem = int(220 * 1024 / (kPlaneSmem<N> + 1024));
  return by_regs < by_smem ? by_regs : by_smem;
}

// forward y and x transforms of one kz plane, times K/Ng, inverse x and y.  kt: K/Ng as [kz][kx][ky].
// The forward transform's code serves y and x in a loop of two, the inverse's x and y: four copies of a
// 64-point transform (74 KB) ran 25% of the issue slots short of instructions.
template <int N>
__global__ void __launch_bounds__(kPlaneThreads<N>, plane_min<N>()) k_xl_plane(Tile t, const double* __restrict__ occ,
                                                              const float* __restrict__ kt, c64* __restrict__ scratch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int C = N * N, PL = planes(N), PITCH = plane_pitch(N);
  constexpr size_t NG = size_t(N) * C;
  static_assert(N % PL == 0 && N % 2 == 0, "planes of a CTA");
  const int a = blockIdx.z, b = blockIdx.y;
  if (t.diag && b < a) return;
  const int team = threadIdx.x / N, x = threadIdx.x - team * N;
  const bool on = team < PL;
  const int z = blockIdx.x * PL + team;
  c64* buf = reinterpret_cast<c64*>(smem_raw + team * plane_stride(N));
  c64* row = buf + x * PITCH;  // this thread's ky
  c64* f = scratch + size_t(a * t.nj + b) * NG + size_t(z) * C + x;
  c64 v[N];
  const bool live = pair_live(t, occ, a, b);
  if (on) sfor<N>([&](auto n) { v[n] = ld_early(f + n * N); });
  if (!live) return;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass) __syncthreads();
    if (!on) continue;
    if (pass)
      sfor<N / 2>([&](auto n) {
        const float4 r = *reinterpret_cast<const float4*>(row + 2 * n);
        v[2 * n] = c64{r.x, r.y};
        v[2 * n + 1] = c64{r.z, r.w};
      });
    Line<N>::forward(v);
    if (pass == 0) {
      sfor<N>([&](auto q) { buf[Line<N>::freq(q) * PITCH + x] = v[q]; });
    } else {
      const float* k = kt + size_t(z) * C + x;  // even in kx: half of the table is read
      sfor<N>([&](auto q) {
        constexpr int kx = Line<N>::freq(q);
        v[q] = v[q] * k[(kx < N - kx ? kx : N - kx) * N];
      });
    }
  }
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (pass) __syncthreads();
    if (!on) continue;
    if (pass) sfor<N>([&](auto q) { v[q] = buf[Line<N>::freq(q) * PITCH + x]; });
    Line<N>::inverse(v);
    if (pass == 0)
      sfor<N / 2>([&](auto n) {
        *reinterpret_cast<float4*>(row + 2 * n) = make_float4(v[2 * n].re, v[2 * n].im, v[2 * n + 1].re, v[2 * n + 1].im);
      });
    else
      sfor<N>([&](auto n) { f[n * N] = v[n]; });
  }
}

// ---- accum ---------------------------------------------------------------------------------

constexpr int OT = 64;  // columns per CTA
// the sum of a line in registers beside the line itself, or (longer lines) in shared memory
constexpr bool sum_in_regs(int n) { return n <= 36; }
template <int N, int S>
constexpr size_t kAccumSmem = (S > 1 || !sum_in_regs(N)) ? size_t(S) * N * OT * sizeof(c64) : 0;
constexpr int accum_min(int n, int s) { return s > 1 ? 1 : n <= 20 ? 10 : n <= 24 ? 8 : 6; }

// W_t -= sum_c d_c partner_c v_c on one column and target per thread; S groups of OT threads share a
// column's sources and add their sums up at the end, in a fixed order.
// Source g ^ k at step k: both targets of a symmetric pair read its field at the same step, so the second
// read hits L2 (64^3, 136 pairs: 168 -> 147 us, DRAM reads 502 -> 356 MB; 24^3, 2080 pairs: 127 -> 88 us).
// k runs down to 0, so a target's own pair, by far its largest term, comes last and the others are summed
// at their own size.
template <int N, int S>
__global__ void __launch_bounds__(OT * S, accum_min(N, S)) k_xl_accum(Tile t, const c64* __restrict__ src,
                                                           const double* __restrict__ occ, const c64* __restrict__ scratch,
                                                           c64* __restrict__ out) {
  using L = Line<N>;
  constexpr int C = N * N, N1 = L::N1, N2 = L::N2;
  constexpr size_t NG = size_t(N) * C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the sources' occupations as floats, NaN for one that is exactly empty (its pair fields may be unwritten): one
  // FP64 conversion per source and CTA, since FP64 instructions issue every 64 cycles on this part
  __shared__ float so[MAXB];
  const bool mir = int(blockIdx.x) >= t.nj;  // the target is one of the tile's sources (mirrored contributions)
  const int g = mir ? blockIdx.x - t.nj : blockIdx.x;
  const int ns = mir ? t.nj : t.ni, s0 = mir ? t.j0 : t.i0, tg = (mir ? t.i0 : t.j0) + g;
  for (int c = threadIdx.x; c < ns; c += OT * S) so[c] = is_zero(occ + s0 + c) ? __int_as_float(0x7fc00000) : float(occ[s0 + c]);
  __syncthreads();
  const int grp = S > 1 ? threadIdx.x / OT : 0, lane = S > 1 ? threadIdx.x % OT : threadIdx.x;
  const int p = blockIdx.y * OT + lane;
  const bool on = C % OT == 0 || p < C;
  c64* sacc = reinterpret_cast<c64*>(smem_raw) + size_t(grp) * (N * OT) + lane;
  c64 acc[sum_in_regs(N) ? N : 1];
  if constexpr (sum_in_regs(N)) sfor<N>([&](auto n) { acc[n] = c64{0.f, 0.f}; });
  else sfor<N>([&](auto n) { sacc[n * OT] = c64{0.f, 0.f}; });
  const c64* sp = src + size_t(s0) * NG + p;
  const c64* vp = scratch + p;
  int span = S;
  while (span < max(t.ni, t.nj)) span *= 2;
  if (on) {
#pragma unroll 1
    for (int k = span - S + grp; k >= 0; k -= S) {
      const int c = g ^ k;
      if (c >= ns) continue;
      const float d = so[c];
      if (isnan(d)) continue;
      const bool cj = mir || (t.diag && c > g);
      const c64* f = vp + size_t(cj ? g * t.nj + c : c * t.nj + g) * NG;
      const c64* w = sp + size_t(c) * NG;
      const float sg = cj ? -d : d;
      c64 v[N];
      sfor<N>([&](auto q) { v[q] = f[L::freq(q) * C]; });
      // the last stage group by group, the partner's points of the next group in flight
      c64 a[2][N1];
      sfor<N1>([&](auto n1) { a[0][n1] = w[L::P::pos(n1, 0) * C]; });
      L::inverse_first(v);
      sfor<N2>([&](auto n2) {
        asm volatile("" ::: "memory");  // keeps the loads of later groups from being hoisted into spills
        constexpr int cur = n2 & 1;
        if constexpr (n2 + 1 < N2) sfor<N1>([&](auto n1) { a[1 - cur][n1] = w[L::P::pos(n1, n2 + 1) * C]; });
        c64 y[N1];
        L::template inverse_group<int(n2)>(v, y);
        sfor<N1>([&](auto n1) {
          constexpr int n = L::P::pos(n1, n2);
          c64 x;
          if constexpr (sum_in_regs(N)) x = acc[n];
          else x = sacc[n * OT];
          const c64 b = a[cur][n1], u = c64{y[n1].re * d, y[n1].im * sg};
          x = rl::padd(x, cmul(b, u));  // one rounding at the sum's size per contribution
          if constexpr (sum_in_regs(N)) acc[n] = x;
          else sacc[n * OT] = x;
        });
      });
    }
  }
  if constexpr (S > 1) {
    if constexpr (sum_in_regs(N)) sfor<N>([&](auto n) { sacc[n * OT] = acc[n]; });
    __syncthreads();
    // the points of the CTA's columns dealt over all its groups
    if (!on) return;
    c64* o = out + size_t(tg) * NG + p;
    const bool zero = !mir && t.first;
    const c64* all = reinterpret_cast<const c64*>(smem_raw) + lane;
    for (int n = grp; n < N; n += S) {
      c64 x = all[n * OT];
#pragma unroll
      for (int s = 1; s < S; ++s) x = x + all[(s * N + n) * OT];
      const c64 r = zero ? c64{0.f, 0.f} : o[n * C];
      o[n * C] = r - x;
    }
  } else {
    if (!on) return;
    c64* o = out + size_t(tg) * NG + p;
    const bool zero = !mir && t.first;
    sfor<N>([&](auto n) {
      c64 x;
      if constexpr (sum_in_regs(N)) x = acc[n];
      else x = sacc[n * OT];
      const c64 r = zero ? c64{0.f, 0.f} : o[n * C];
      o[n * C] = r - x;
    });
  }
}

template <int N, int S>
void run_accum(const Tile& t, const c64* src, const double* occ, const c64* scratch, c64* out, cudaStream_t st) {
  static DeviceOnce once;
  once([] {
    PT_CUDA_CHECK(
        cudaFuncSetAttribute(k_xl_accum<N, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kAccumSmem<N, S>)));
  });
  const int targets = t.nj + (t.sym && !t.diag ? t.ni : 0);
  PT_LAUNCH((k_xl_accum<N, S>), dim3(targets, (N * N + OT - 1) / OT), OT * S, (kAccumSmem<N, S>), st, t, src, occ, scratch,
            out);
}

template <int N>
void run_tile(const Tile& t, const c64* src, const c64* tgt, const double* occ, const float* kt, c64* scratch, c64* out,
              int sms, cudaStream_t st) {
  static DeviceOnce once;
  once([] {
    PT_CUDA_CHECK(cudaFuncSetAttribute(k_xl_plane<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kPlaneSmem<N>)));
  });
  constexpr int C = N * N;
  PT_LAUNCH(k_xl_zfwd<N>, dim3((C + ZT - 1) / ZT, t.nj, t.ni), ZT, 0, st, t, src, tgt, occ, scratch);
  PT_LAUNCH(k_xl_plane<N>, dim3(N / planes(N), t.nj, t.ni), kPlaneThreads<N>, kPlaneSmem<N>, st, t, occ, kt, scratch);
  const int targets = t.nj + (t.sym && !t.diag ? t.ni : 0), warps = targets * ((C + OT - 1) / OT) * (OT / 32);
  // four groups per column where one leaves fewer than 6 warps to an SM (24^3 N = 16: 42 against 48 us a call; at 9
  // warps, 36^3 N = 32, 212 against 205)
  if (warps < 6 * sms) run_accum<N, 4>(t, src, occ, scratch, out, st);
  else run_accum<N, 1>(t, src, occ, scratch, out, st);
}

}  // namespace

bool exchange_lines_applies(const pt_ctx* ctx, const pt_grid& g) {
  return fixed_cubic(g) && (exchange64_applies(g) ? ctx->exchange64_engine == 0 : ctx->exchange64_engine != 1);
}

long long exchange_lines(pt_ctx* ctx, const c64* src, const double* occ, int N, const c64* tgt, int M, bool sym, c64* out,
                         const pt_grid& g, const pt_kernel& k, size_t budget, cudaStream_t st) {
  const size_t field = ng_of(g) * sizeof(c64);
  int B = int(std::floor(std::sqrt(double(std::max<size_t>(1, budget / field)))));
  B = std::max(1, std::min({B, std::max(N, M), MAXB}));
  pt_grid gt = g;  // the plane pass reads K with ky fastest: the table of the cell with Lx and Ly exchanged
  std::swap(gt.L[0], gt.L[1]);
  const float* kt = static_cast<const float*>(kernel_table(ctx, gt, k, PT_FP32));
  c64* scratch = static_cast<c64*>(
      ctx->get(ctx->tagged("exchange_scratch"), size_t(std::min(B, N)) * size_t(std::min(B, M)) * field));
  const int nb = (N + B - 1) / B, mb = (M + B - 1) / B;
  for (int J = 0; J < mb; ++J)
    for (int I = 0; I < (sym ? J + 1 : nb); ++I) {
      const Tile t{I * B, std::min(B, N - I * B), J * B, std::min(B, M - J * B), int(sym), int(sym && I == J), int(I == 0)};
      switch (g.nx) {
#define PT_CASE(n)                                                     \
  case n:                                                              \
    run_tile<n>(t, src, tgt, occ, kt, scratch, out, ctx->num_sms, st); \
    break;
        PT_FIXED_SIZES(PT_CASE)
#undef PT_CASE
        default:
          fail(PT_INVALID_ARG, "no compile-time FFT kernels for this grid side");
      }
    }
  return sym ? (long long)N * (N + 1) / 2 : (long long)N * M;
}

}  // namespace pt
