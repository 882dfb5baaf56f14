// Line kernels of the FP32 exchange (exchange_lines.cu has the method and its measurements): the passes
// along z, shared by the translation units of the cubic and the other grids.
#pragma once

#include <algorithm>

#include "exchange_sched.h"
#include "fft_reg.cuh"
#include "internal.h"

namespace pt {

// One tile of the pair schedule: sources i0 .. i0 + ni, targets j0 .. j0 + nj, the field of pair
// (i0 + a, j0 + b) in slot a nj + b.  In the symmetric case a diagonal tile (diag) holds the pairs
// a <= b, and the pairs of an off-diagonal tile feed both their orbitals.  first: the tile's
// targets have no earlier tile.
struct Tile {
  int i0, ni, j0, nj, sym, diag, first;
};

// axis lengths with line kernels (a grid of others, or of shorter axes, runs the general kernels)
#define PT_LINE_SIZES(X) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64)
bool line_length(int n);

// one tile on a grid that is not cubic (exchange_lines_axes.cu)
void exchange_tile_axes(const pt_grid& g, const Tile& t, const c64* src, const c64* tgt, const double* occ, const float* kt,
                        c64* scratch, c64* out, int sms, cudaStream_t st);

namespace {

using rl::Line;
using rl::sfor;

constexpr int MAXB = 128;  // largest pair-tile side

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

// rho = conj(src_i) tgt_j on one column, forward z transform (CC: the columns of the grid, 0 if given at run time)
template <int N, int CC>
__global__ void __launch_bounds__(ZT, zmin(N)) k_xl_zfwd(Tile t, const c64* __restrict__ src, const c64* __restrict__ tgt,
                                                         const double* __restrict__ occ, c64* __restrict__ scratch,
                                                         int columns) {
  const int C = CC ? CC : columns;
  const size_t NG = size_t(N) * C;
  const int a = blockIdx.z, b = blockIdx.y;
  if (t.diag && b < a) return;
  const int p = blockIdx.x * ZT + threadIdx.x;
  if ((CC == 0 || CC % ZT) && p >= C) return;
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

// ---- accum ---------------------------------------------------------------------------------

// Tensor memory as per-thread storage: a thread of warp w of a 128-thread CTA owns row 32 w + lane of the columns that
// the CTA allocated, and moves words of its row by index.
constexpr int TM_COLS = 128;  // words per thread: a line of 64 complex numbers

// words [a, a + W) of the thread's row (a: row and column address) to r; the values may be used after tm_loaded
template <int W>
__device__ __forceinline__ void tm_load(uint32_t a, float* r) {
  if constexpr (W >= 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
          "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(a));
    if constexpr (W > 16) tm_load<W - 16>(a + 16, r + 16);
  } else if constexpr (W >= 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7])
                 : "r"(a));
    if constexpr (W > 8) tm_load<W - 8>(a + 8, r + 8);
  } else if constexpr (W >= 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3])
                 : "r"(a));
    if constexpr (W > 4) tm_load<W - 4>(a + 4, r + 4);
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=f"(r[0]), "=f"(r[1]) : "r"(a));
  }
}
// the loads of r have arrived (the empty statements keep its uses behind the wait)
template <int W>
__device__ __forceinline__ void tm_loaded(float* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  sfor<W>([&](auto i) { asm volatile("" : "+f"(r[i])); });
}
template <int W>
__device__ __forceinline__ void tm_store(uint32_t a, const float* r) {
  if constexpr (W >= 16) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(a),
        "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]),
        "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
        : "memory");
    if constexpr (W > 16) tm_store<W - 16>(a + 16, r + 16);
  } else if constexpr (W >= 8) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(a), "f"(r[0]), "f"(r[1]),
                 "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7])
                 : "memory");
    if constexpr (W > 8) tm_store<W - 8>(a + 8, r + 8);
  } else if constexpr (W >= 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(r[0]), "f"(r[1]), "f"(r[2]),
                 "f"(r[3])
                 : "memory");
    if constexpr (W > 4) tm_store<W - 4>(a + 4, r + 4);
  } else {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(a), "f"(r[0]), "f"(r[1]) : "memory");
  }
}
__device__ __forceinline__ void tm_stored() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Where a line's sum lives beside the line itself: in registers (short lines), in tensor memory (64 points: its groups of
// eight move 16 words at a time, and the kernel was waiting on the shared-memory queue: 147 -> 105 us for 136 pairs,
// one application at N = 96 10.9 -> 9.65 ms), else in shared memory (tensor memory moves groups of 3 to 6 points in
// pieces and needs 128 columns to a CTA: 60^3 N = 64 3.5 -> 3.9 ms, 40^3, 48^3 and 54^3 unchanged; registers for
// the sum as well leave fewer warps: 32^3 N = 96 1.16 against 1.08 ms, 36^3 1.73 against 1.68).
constexpr bool sum_in_regs(int n) { return n <= 20; }
constexpr bool sum_in_tmem(int n, int s) { return n == 64 && s == 1; }
constexpr int accum_columns(int n, int s) { return sum_in_tmem(n, s) ? 128 : 64; }  // per CTA
template <int N, int S>
constexpr size_t kAccumSmem =
    (S > 1 || !(sum_in_regs(N) || sum_in_tmem(N, S))) ? size_t(S) * N * accum_columns(N, S) * sizeof(c64) : 0;
constexpr int accum_min(int n, int s) { return s > 1 ? 1 : n <= 24 ? 10 : n <= 32 ? 8 : sum_in_tmem(n, s) ? 3 : 6; }

// W_t -= sum_c d_c partner_c v_c on one column and target per thread; S groups of threads share a column's sources and
// add their sums up at the end, in a fixed order.
// Source g ^ k at step k: both targets of a symmetric pair read its field at the same step, so the second
// read hits L2 (64^3, 136 pairs: 168 -> 147 us, DRAM reads 502 -> 356 MB; 24^3, 2080 pairs: 127 -> 88 us).
// k runs down to 0, so a target's own pair, by far its largest term, comes last and the others are summed
// at their own size.
template <int N, int CC, int S>
__global__ void __launch_bounds__(accum_columns(N, S) * S, accum_min(N, S))
    k_xl_accum(Tile t, const c64* __restrict__ src, const double* __restrict__ occ, const c64* __restrict__ scratch,
               c64* __restrict__ out, int columns) {
  using L = Line<N>;
  constexpr int N1 = L::N1, N2 = L::N2, OT = accum_columns(N, S);
  constexpr bool regs = sum_in_regs(N), tmem = sum_in_tmem(N, S);
  const int C = CC ? CC : columns;
  const size_t NG = size_t(N) * C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // the sources' occupations as floats: one FP64 conversion per source and CTA, since FP64 instructions issue every 64
  // cycles on this part
  __shared__ float so[MAXB];
  __shared__ uint32_t tm_holder;
  const bool mir = int(blockIdx.x) >= t.nj;  // the target is one of the tile's sources (mirrored contributions)
  const int g = mir ? blockIdx.x - t.nj : blockIdx.x;
  const int ns = mir ? t.nj : t.ni, s0 = mir ? t.j0 : t.i0, tg = (mir ? t.i0 : t.j0) + g;
  for (int c = threadIdx.x; c < ns; c += OT * S) so[c] = float(occ[s0 + c]);
  uint32_t row = 0;  // address of the thread's row in tensor memory
  if constexpr (tmem) {
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       unsigned(__cvta_generic_to_shared(&tm_holder))),
                   "r"(TM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if constexpr (tmem) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    row = tm_holder + ((threadIdx.x & ~31u) << 16);
    float zero[2 * N1];
    sfor<2 * N1>([&](auto i) { zero[i] = 0.f; });
    sfor<N2>([&](auto n2) { tm_store<2 * N1>(row + n2 * (2 * N1), zero); });
    tm_stored();
  }
  const int grp = S > 1 ? threadIdx.x / OT : 0, lane = S > 1 ? threadIdx.x % OT : threadIdx.x;
  const int p = blockIdx.y * OT + lane;
  const bool on = (CC && CC % OT == 0) || p < C;
  const int pc = on ? p : C - 1;  // tensor memory is moved by whole warps: lanes past the last column run along
  c64* sacc = reinterpret_cast<c64*>(smem_raw) + size_t(grp) * (N * OT) + lane;
  c64 acc[regs ? N : 1];
  if constexpr (regs) sfor<N>([&](auto n) { acc[n] = c64{0.f, 0.f}; });
  else if constexpr (!tmem) sfor<N>([&](auto n) { sacc[n * OT] = c64{0.f, 0.f}; });
  const c64* sp = src + size_t(s0) * NG + pc;
  const c64* vp = scratch + pc;
  int span = S;
  while (span < max(t.ni, t.nj)) span *= 2;
#pragma unroll 1
  for (int k = (tmem || on) ? span - S + grp : -1; k >= 0; k -= S) {
    const int c = g ^ k;
    if (c >= ns) continue;
    const float d = so[c];
    if (d == 0.f) continue;  // empty: its pair fields may be unwritten (a NaN is not, and belongs to the result)
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
      [[maybe_unused]] float x[2 * N1];  // the sums of the group's points
      if constexpr (tmem) tm_load<2 * N1>(row + n2 * (2 * N1), x);
      c64 y[N1];
      L::template inverse_group<int(n2)>(v, y);
      if constexpr (tmem) tm_loaded<2 * N1>(x);
      sfor<N1>([&](auto n1) {
        constexpr int n = L::P::pos(n1, n2);
        c64 s;
        if constexpr (regs) s = acc[n];
        else if constexpr (tmem) s = c64{x[2 * n1], x[2 * n1 + 1]};
        else s = sacc[n * OT];
        // one rounding at the sum's size per contribution
        s = rl::padd(s, cmul(a[cur][n1], c64{y[n1].re * d, y[n1].im * sg}));
        if constexpr (regs) acc[n] = s;
        else if constexpr (tmem) {
          x[2 * n1] = s.re;
          x[2 * n1 + 1] = s.im;
        } else sacc[n * OT] = s;
      });
      if constexpr (tmem) tm_store<2 * N1>(row + n2 * (2 * N1), x);
    });
    if constexpr (tmem) tm_stored();
  }
  c64* o = out + size_t(tg) * NG + pc;
  const bool zero = !mir && t.first;
  if constexpr (S > 1) {
    if constexpr (regs) sfor<N>([&](auto n) { sacc[n * OT] = acc[n]; });
    __syncthreads();
    // the points of the CTA's columns dealt over all its groups
    if (!on) return;
    const c64* all = reinterpret_cast<const c64*>(smem_raw) + lane;
    for (int n = grp; n < N; n += S) {
      c64 x = all[n * OT];
#pragma unroll
      for (int s = 1; s < S; ++s) x = x + all[(s * N + n) * OT];
      const c64 r = zero ? c64{0.f, 0.f} : o[n * C];
      o[n * C] = r - x;
    }
  } else if constexpr (tmem) {
    sfor<N2>([&](auto n2) {
      float x[2 * N1];
      tm_load<2 * N1>(row + n2 * (2 * N1), x);
      tm_loaded<2 * N1>(x);
      sfor<N1>([&](auto n1) {
        constexpr int n = L::P::pos(n1, n2);
        if (on) o[n * C] = (zero ? c64{0.f, 0.f} : o[n * C]) - c64{x[2 * n1], x[2 * n1 + 1]};
      });
    });
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_holder), "r"(TM_COLS) : "memory");
    }
  } else {
    if (!on) return;
    sfor<N>([&](auto n) {
      c64 x;
      if constexpr (regs) x = acc[n];
      else x = sacc[n * OT];
      const c64 r = zero ? c64{0.f, 0.f} : o[n * C];
      o[n * C] = r - x;
    });
  }
}

template <int N, int CC, int S>
void launch_accum(const Tile& t, const c64* src, const double* occ, const c64* scratch, c64* out, int C, cudaStream_t st) {
  static DeviceOnce once;
  once([] {
    PT_CUDA_CHECK(
        cudaFuncSetAttribute(k_xl_accum<N, CC, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kAccumSmem<N, S>)));
  });
  constexpr int OT = accum_columns(N, S);
  const int targets = t.nj + (t.sym && !t.diag ? t.ni : 0);
  PT_LAUNCH((k_xl_accum<N, CC, S>), dim3(targets, (C + OT - 1) / OT), OT * S, (kAccumSmem<N, S>), st, t, src, occ, scratch,
            out, C);
}

template <int N, int CC>
void run_zfwd(const Tile& t, const c64* src, const c64* tgt, const double* occ, c64* scratch, int C, cudaStream_t st) {
  PT_LAUNCH((k_xl_zfwd<N, CC>), dim3((C + ZT - 1) / ZT, t.nj, t.ni), ZT, 0, st, t, src, tgt, occ, scratch, C);
}

template <int N, int CC>
void run_accum(const Tile& t, const c64* src, const double* occ, const c64* scratch, c64* out, int C, int sms,
               cudaStream_t st) {
  const int targets = t.nj + (t.sym && !t.diag ? t.ni : 0), warps = targets * ((C + 63) / 64) * 2;
  // four groups per column where one leaves fewer than 6 warps to an SM (24^3 N = 16: 42 against 48 us a call; at 9
  // warps, 36^3 N = 32, 212 against 205)
  if (warps < 6 * sms) launch_accum<N, CC, 4>(t, src, occ, scratch, out, C, st);
  else launch_accum<N, CC, 1>(t, src, occ, scratch, out, C, st);
}

}  // namespace

}  // namespace pt
