// Wide-tile Gram contractions on the 5th-generation tensor cores (tcgen05, TF32 inputs):
//   C0 = scale * A^H B0   and, optionally in the same pass,   C1 = scale * A^H B1
// with A, B0, B1 complex64, orbital-major (each orbital a K-major row of K' = 2 Ng interleaved
// floats).  The overlap S = <Phi|Phi> and the subspace matrix <Phi|H Phi> of the PT-IM inner
// iteration (Sec. IV-A2) share their left operand, so one pass computes both.
//
// A tile is one 64-orbital block of A against two 64-orbital B halves: the MMA is M = 128 (rows
// 0..63 the A orbitals, 64..127 the same orbitals times i, giving Re and Im of A^H B in one real
// GEMM, as in the 64 x 64 kernel) by N = 128 (half 0 and half 1, each from B0 or B1).  The wider N
// halves the tensor-core operand traffic and the A-side conversion per product compared with
// N = 64 tiles, and the shared A block is converted once for both halves.  The FP32 accuracy
// comes from three TF32 products hi*hi + hi*lo + lo*hi (the raw FP32 value is its own TF32 "hi";
// "lo" = x - tf32(x) is written by the converter warps).
//
// Warp roles (640 threads, five warpgroups): one lane of group 0 issues tcgen05.mma; groups 1 and 2 take the
// stages in turn: they copy them (cp.async), write [A; i A] as hi and lo parts into TMEM, where the MMA reads its A
// operand, and B's lo parts into shared memory; groups 3 and 4 read the accumulator out every `period` stages
// into Kahan-compensated FP32 registers, 64 of its 128 columns each.  Two TMEM accumulators alternate; setmaxnreg
// gives the readout the registers that the other groups do without.
//   What bounds it: a stage of three products is 770 cycles of MMA, 380 of B operand reads and 600 of copies,
// conversions and spills on the shared-memory pipe, and takes about 1450; without two of the three products it took
// 1200, without the conversions or the copies 1400, without most of the readout 1300 (no single one is the wall).  Before, with
// one TMA-fed ring of 64 KB stages, A in shared memory and 16 warps that converted and read out in turn, it took
// 1950: boxes of 64 rows of 128 bytes arrive at no more than 31 GB/s a CTA (1500 cycles a stage), A operands
// were another 380 cycles of reads, and conversion and readout waited for each other.  54^3, 200 x 200: 625 -> 477 us
// a call, 64^3, 320 x 320 1776 -> 1354, its Hermitian form 1148 -> 884.  A in TMEM alone gave nothing (54^3: 690 in place
// of 670); a third converter group costs the readout registers (541 against 520), four readout groups of 32
// columns likewise (562 against 539).
// The K range of every tile is split over CTAs; each CTA writes an FP64 partial tile and a
// reduction kernel sums the splits into C0/C1, mirroring the blocks of a Hermitian product that
// no tile computed.  Every mbarrier wait is bounded (%globaltimer): on expiry the CTA records an
// error, leaves its loops, waits for its own copies and MMAs and frees its TMEM.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "packed.cuh"
#include "split_sum.cuh"
#include "tma.cuh"

namespace pt {

namespace {

constexpr int WB = 64;                    // orbitals per A block and per B half
constexpr int WN = 2 * WB;                // MMA N
constexpr int WK = 32;                    // floats of K per stage (one 128-byte swizzled row)
constexpr int W_CVT = 128;                // threads of one converter warpgroup
constexpr int W_RO = 256;                 // readout threads
constexpr int W_THREADS = 128 + 2 * W_CVT + W_RO;
constexpr uint32_t ROWS = 64 * 128;       // 64 rows of one 128-byte stage row
// shared memory: a ring of raw stages [A][half 0 | half 1] (the raw B is the "hi" operand) and one of
// [half 0 lo | half 1 lo]
constexpr int RAW = 6, LO = 4;
constexpr uint32_t RAW_BYTES = 3 * ROWS, LO_BYTES = 2 * ROWS;
constexpr uint32_t OFF_LO = RAW * RAW_BYTES;
constexpr uint32_t OFF_BAR = OFF_LO + LO * LO_BYTES;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 256 + 1024;
// TMEM columns: two accumulators, then a ring of LO converted A stages (hi and lo)
constexpr int A_COL0 = 2 * WN;
constexpr int TMEM_COLS = 512;
static_assert(A_COL0 + LO * 2 * WK <= TMEM_COLS, "TMEM columns");
constexpr int AHEAD = 2;                  // stages of its own that a converter warpgroup has in flight
static_assert(RAW == 2 * AHEAD + 2 && LO == 4, "the slots that the stage two back frees");
// registers a thread: 640 threads start with 96; MMA 24, converters 48, readout 176 (472 of 480 a lane of each group)
constexpr int R_MMA = 24, R_CVT = 48, R_RO = 176;
static_assert(R_MMA + 2 * R_CVT + 2 * R_RO <= 5 * 96, "register split");
constexpr uint64_t TIMEOUT_NS = 2000000000ull;

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  // K-major, 128B swizzle: start >> 4, LBO unused (1), SBO = 1024 B between 8-row groups,
  // fixed 0b001 at bits 46..48, swizzle mode 2 (128B) at bits 61..63
  uint64_t d = uint64_t((addr >> 4) & 0x3FFFu);
  d |= uint64_t(1) << 16;
  d |= uint64_t(1024 >> 4) << 32;
  d |= uint64_t(1) << 46;
  d |= uint64_t(2) << 61;
  return d;
}

// instruction descriptor: D f32, A/B tf32, both K-major, N = 128, M = 128
constexpr uint32_t IDESC_W = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(WN >> 3) << 17) | (uint32_t(128 >> 4) << 24);

// A from TMEM (128 lanes by 8 columns), B from shared memory
__device__ __forceinline__ void mma_w(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(IDESC_W), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void commit_w(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// 8 columns of this warp's TMEM lanes
__device__ __forceinline__ void st8(uint32_t taddr, float4 a, float4 b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
               "r"(__float_as_uint(a.x)), "r"(__float_as_uint(a.y)), "r"(__float_as_uint(a.z)), "r"(__float_as_uint(a.w)),
               "r"(__float_as_uint(b.x)), "r"(__float_as_uint(b.y)), "r"(__float_as_uint(b.z)), "r"(__float_as_uint(b.w))
               : "memory");
}
__device__ __forceinline__ void wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float tf32_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }
// 16-byte shared-memory accesses by 32-bit shared-window address
__device__ __forceinline__ float4 lds128(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ float4 hi4(float4 v) { return make_float4(tf32_hi(v.x), tf32_hi(v.y), tf32_hi(v.z), tf32_hi(v.w)); }
__device__ __forceinline__ float4 lo4(float4 v) {
  const c64 a = rl::psub(c64{v.x, v.y}, c64{tf32_hi(v.x), tf32_hi(v.y)});
  const c64 b = rl::psub(c64{v.z, v.w}, c64{tf32_hi(v.z), tf32_hi(v.w)});
  return make_float4(a.re, a.im, b.re, b.im);
}
__device__ __forceinline__ float4 times_i(float4 v) { return make_float4(-v.y, v.x, -v.w, v.z); }

// one tile: A block r against half 0 = block c0 of B(m0) and half 1 = block c1 of B(m1)
struct WideTile {
  int r, m0, c0, m1, c1;
};

struct WideArgs {
  const float *A, *B0, *B1;
  int N1, N2;
  int row;  // floats of an orbital
  int stages_total;
  int stages_per_split;
  int split3;
  int period;
};

// 16 bytes from global to shared memory, the bytes from `bytes` on as zeros
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// barrier 1 + g of one converter warpgroup; whether every thread brought `ok`
__device__ __forceinline__ bool group_all(int g, bool ok) {
  int r;
  if (g == 0)
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, 128, p;\n selp.s32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(int(ok))
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n barrier.cta.red.and.pred q, 2, 128, p;\n selp.s32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(int(ok))
        : "memory");
  return r != 0;
}

__global__ void __launch_bounds__(W_THREADS, 1)
    k_gram_tc_wide(const WideTile* __restrict__ tiles, WideArgs P, double* __restrict__ part, int* __restrict__ err) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  const uint32_t bar0 = base + OFF_BAR;
  auto bar_cvt = [&](int it) { return bar0 + 8u * (it % RAW); };
  auto bar_empty = [&](int it) { return bar0 + 8u * (RAW + it % RAW); };
  auto bar_acc_full = [&](int b) { return bar0 + 8u * (2 * RAW + b); };
  auto bar_acc_empty = [&](int b) { return bar0 + 8u * (2 * RAW + 2 + b); };
  const uint32_t bar_drain = bar0 + 8u * (2 * RAW + 4);
  volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(sm + OFF_BAR + 192);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(sm + OFF_BAR + 200);
  auto raw_stage = [&](int it) { return base + uint32_t(it % RAW) * RAW_BYTES; };
  auto lo_stage = [&](int it) { return base + OFF_LO + uint32_t(it % LO) * LO_BYTES; };
  auto a_cols = [&](int it) { return uint32_t(A_COL0 + (it % LO) * 2 * WK); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, group = tid >> 7;
  const int tile = blockIdx.x, split = blockIdx.y;
  const int st0 = split * P.stages_per_split;
  const int st1 = min(P.stages_total, st0 + P.stages_per_split);
  const int nst = max(0, st1 - st0);
  const int period = P.period;
  const int nper = (nst + period - 1) / period;

  if (tid == 0) {
    for (int s = 0; s < RAW; ++s) {
      mbar_init(bar_cvt(s), W_CVT);
      mbar_init(bar_empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_acc_full(b), 1);
      mbar_init(bar_acc_empty(b), W_RO);
    }
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + OFF_BAR + 192),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_holder;
  auto fail_out = [&](int code) {
    atomicOr(err, code);
    *abort_flag = 1;
  };

  if (group == 0) {
    // ---------------- MMA issuer (one lane) ----------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_MMA));
    if (tid == 0) {
      for (int it = 0; it < nst && !*abort_flag; ++it) {
        const int per = it / period, b = per & 1;
        if (it % period == 0 && per >= 2 && !mbar_wait(bar_acc_empty(b), ((per / 2) - 1) & 1, TIMEOUT_NS)) {
          fail_out(2);
          break;
        }
        if (!mbar_wait(bar_cvt(it), (it / RAW) & 1, TIMEOUT_NS)) {
          fail_out(4);
          break;
        }
        fence_after();
        const uint32_t d = tmem + uint32_t(b * WN);
        const uint32_t ahi = tmem + a_cols(it), alo = ahi + WK;
        const uint32_t bhi = raw_stage(it) + ROWS, blo = lo_stage(it);
#pragma unroll
        for (int kk = 0; kk < WK / 8; ++kk) {
          const uint32_t off = uint32_t(kk * 32);
          const uint32_t first = (it % period == 0 && kk == 0) ? 0u : 1u;
          mma_w(d, ahi + 8 * kk, desc_sw128(bhi + off), first);
          if (P.split3) {
            mma_w(d, ahi + 8 * kk, desc_sw128(blo + off), 1u);
            mma_w(d, alo + 8 * kk, desc_sw128(bhi + off), 1u);
          }
        }
        commit_w(bar_empty(it));
        if (it % period == period - 1 || it == nst - 1) commit_w(bar_acc_full(b));
      }
      // all issued MMAs complete before TMEM is freed
      commit_w(bar_drain);
      if (!mbar_wait(bar_drain, 0, TIMEOUT_NS)) atomicOr(err, 256);
    }
    __syncwarp();
  } else if (group <= 2) {
    // ---------------- converters: warpgroup g takes the stages of its parity ----------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_CVT));
    const int g = group - 1, ct = tid & 127;
    const WideTile T = tiles[tile];
    // copies: chunk ct & 7 (16 bytes) of the rows (ct >> 3) + 16 j of A (j < 4) and of the halves (4 each); a row's
    // chunks are swizzled by its index mod 8, which is that of ct >> 3
    const int crow = ct >> 3;
    const uint32_t cdst = uint32_t(crow) * 128u + uint32_t((ct & 7) ^ (crow & 7)) * 16u;
    const size_t row16 = size_t(16) * P.row;
    const int ra = T.r * WB + crow, rb = T.c0 * WB + crow;
    // Rows past a matrix, and an absent second half, are not copied: whatever their shared memory holds reaches only
    // accumulator entries that are never reduced.
    const bool two = T.m1 >= 0;
    const int rc = two ? T.c1 * WB + crow : P.N2;
    const float* const pb = T.m0 == 1 ? P.B1 : P.B0;
    const float* const pc = T.m1 == 1 ? P.B1 : P.B0;
    const int na = (P.N1 - ra + 15) / 16, nb = (P.N2 - rb + 15) / 16, nc = (P.N2 - rc + 15) / 16;
    const int kc = 4 * (ct & 7);
    const float* const qa = P.A + size_t(ra) * P.row + kc;
    const float* const qb = pb + size_t(rb) * P.row + kc;
    const float* const qc = pc + size_t(rc) * P.row + kc;
    auto copy = [&](int it) {
      const uint32_t dst = raw_stage(it) + cdst;
      const int k = (st0 + it) * WK;
      // a row's end: a chunk is in it whole or not at all (rows are a multiple of four floats), zeros in its place
      const int bytes = k + kc < P.row ? 16 : 0;
      const int kin = bytes ? k : -kc;
      auto rows4 = [&](const float* q, int n, uint32_t d) {
#pragma unroll
        for (int j = 0; j < 4; ++j, q += row16)
          if (j < n) cp16(d + uint32_t(j) * 2048u, q, bytes);
      };
      rows4(qa + kin, na, dst);
      rows4(qb + kin, nb, dst + ROWS);
      rows4(qc + kin, nc, dst + 2 * ROWS);
    };
    auto commit_copies = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    for (int n = 0; n < AHEAD; ++n) {
      if (g + 2 * n < nst) copy(g + 2 * n);
      commit_copies();
    }
    // A: this thread's TMEM lane ct is row ct of the MMA's A: orbital row ct & 63, times i from 64 on
    const int arow = ct & (WB - 1), sw = arow & 7;
    const bool imag = ct >= WB;
    const uint32_t lane_base = uint32_t(32 * (warp & 3)) << 16;
    for (int it = g; it < nst; it += 2) {
      const bool ok = *abort_flag == 0;
      asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
      if (!group_all(g, ok)) break;  // every thread's copies of the stage are there
      fence_after();
      const uint32_t st = raw_stage(it);
      const uint32_t at = tmem + lane_base + a_cols(it);
      const uint32_t ast = st + uint32_t(arow) * 128u;
      auto rows_a = [&](auto turn) {
#pragma unroll
        for (int c = 0; c < 8; c += 2) {
          const float4 r0 = lds128(ast + uint32_t(c ^ sw) * 16u), r1 = lds128(ast + uint32_t((c + 1) ^ sw) * 16u);
          const float4 a0 = turn ? times_i(r0) : r0, a1 = turn ? times_i(r1) : r1;
          st8(at + 4 * c, hi4(a0), hi4(a1));
          if (P.split3) st8(at + WK + 4 * c, lo4(a0), lo4(a1));
        }
      };
      if (imag)
        rows_a(std::true_type{});
      else
        rows_a(std::false_type{});
      if (P.split3) {
        // a lo chunk has the swizzled position of its raw one
        const uint32_t src = st + ROWS + uint32_t(ct) * 16u, dst = lo_stage(it) + uint32_t(ct) * 16u;
#pragma unroll
        for (int j = 0; j < 8; ++j) sts128(dst + 2048u * j, lo4(lds128(src + 2048u * j)));
      }
      wait_st();
      fence_before();
      fence_proxy_async_smem();
      mbar_arrive(bar_cvt(it));
      // once the stage two back is multiplied its raw slot takes the copy for it + 2 AHEAD (RAW = 2 AHEAD + 2), and its
      // slots in shared memory and TMEM (LO = 4) the next conversion
      if (it >= 2 && !mbar_wait(bar_empty(it - 2), ((it - 2) / RAW) & 1, TIMEOUT_NS)) fail_out(16);
      if (it + 2 * AHEAD < nst) copy(it + 2 * AHEAD);
      commit_copies();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ---------------- readout: warpgroup h owns the accumulator columns [64 h, 64 h + 64) ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R_RO));
    const int h = group - 3, quad = warp & 3;
    const uint32_t lane_base = uint32_t(32 * quad) << 16;
    c64 sum[32], comp[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) sum[c] = comp[c] = c64{0.f, 0.f};
    // waits and aborts are decided per warp (vote), so the .sync.aligned TMEM loads run converged
    for (int per = 0; per < nper; ++per) {
      const int b = per & 1;
      if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
      if (!__all_sync(0xffffffffu, mbar_wait(bar_acc_full(b), (per / 2) & 1, TIMEOUT_NS))) {
        fail_out(32);
        break;
      }
      fence_after();
#pragma unroll
      for (int c0 = 0; c0 < 64; c0 += 8) {
        float v[8];
        ld8(tmem + lane_base + uint32_t(b * WN + 64 * h + c0), v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = c0 / 2 + i;
          const c64 y = rl::psub(c64{v[2 * i], v[2 * i + 1]}, comp[c]);
          const c64 t = rl::padd(sum[c], y);
          comp[c] = rl::psub(rl::psub(t, sum[c]), y);
          sum[c] = t;
          // added up before the next columns are loaded: eight loads in flight would hold 64 registers
          asm volatile("" : "+f"(sum[c].re), "+f"(sum[c].im), "+f"(comp[c].re), "+f"(comp[c].im)::"memory");
        }
      }
      fence_before();
      mbar_arrive(bar_acc_empty(b));
    }
    // FP64 partial: rows 0..63 real part, 64..127 imaginary part; columns 0..63 half 0, 64..127 half 1
    const int row = 32 * quad + lane;
    double* out = part + ((size_t(split) * gridDim.x + tile) * 128 + row) * WN + 64 * h;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const double2 v = make_double2(double(sum[c].re) - double(comp[c].re), double(sum[c].im) - double(comp[c].im));
      asm volatile("st.global.v2.f64 [%0], {%1, %2};" ::"l"(out + 2 * c), "d"(v.x), "d"(v.y) : "memory");
    }
  }
  // teardown: every role has left its loop; free TMEM
  fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// C_m[i][j] = scale * sum_split part[split][tile][row][col] through a block lookup: entry
// (m, i / 64, j / 64) = tile * 4 + half * 2 + mirror (-1: not computed); a mirrored block is the
// conjugate transpose of block (j / 64, i / 64)
template <int G>
__global__ void __launch_bounds__(SUM_THREADS) k_gram_tc_wide_reduce(const double* __restrict__ part, int nsplit, int ntiles,
                                                                     const int* __restrict__ lut, int nbi, int nbj, int N1,
                                                                     int N2, double scale, c128* __restrict__ C0,
                                                                     c128* __restrict__ C1) {
  const size_t e = split_entry<G>();
  const int m = int(blockIdx.y);
  const bool in = e < size_t(N1) * N2;
  c128* C = m == 0 ? C0 : C1;
  int i = int(e / N2), j = int(e % N2);
  const int code = in ? lut[(size_t(m) * nbi + i / WB) * nbj + j / WB] : -1;
  const int tile = code >> 2, half = (code >> 1) & 1, mirror = code & 1;
  if (mirror) {
    const int t = i;
    i = j;
    j = t;
  }
  const int r = i % WB, c = half * WB + j % WB;
  double re, im;
  const bool owner = split_sum<G>(
      nsplit, code >= 0,
      [&](int s) {
        const double* p = part + (size_t(s) * ntiles + tile) * 128 * WN;
        return c128{p[size_t(r) * WN + c], p[size_t(WB + r) * WN + c]};
      },
      re, im);
  if (owner) C[e] = mirror ? c128{re * scale, -im * scale} : c128{re * scale, im * scale};
}

struct WidePlan {
  int ntiles = 0;
  WideTile* tiles = nullptr;  // device
  int* lut = nullptr;         // device, 2 x nbi x nbj
  ~WidePlan() {
    cudaFree(tiles);
    cudaFree(lut);
  }
};

std::shared_ptr<WidePlan> wide_plan(pt_ctx* ctx, int N1, int N2, bool two, bool herm) {
  char key[96];
  snprintf(key, sizeof(key), "gram_wide:%d:%d:%d:%d", N1, N2, int(two), int(herm));
  auto it = ctx->caches.find(key);
  if (it != ctx->caches.end()) return std::static_pointer_cast<WidePlan>(it->second);
  const int nbi = (N1 + WB - 1) / WB, nbj = (N2 + WB - 1) / WB;
  std::vector<WideTile> tl;
  std::vector<int> lut(size_t(2) * nbi * nbj, -1);
  auto put = [&](int m, int r, int c, int t, int half) {
    lut[(size_t(m) * nbi + r) * nbj + c] = t * 4 + half * 2;
    if (herm && r != c) lut[(size_t(m) * nbi + c) * nbj + r] = t * 4 + half * 2 + 1;
  };
  for (int r = 0; r < nbi; ++r) {
    std::vector<int> cs;
    for (int c = herm ? r : 0; c < nbj; ++c) cs.push_back(c);
    if (two) {
      for (int c : cs) {
        const int t = int(tl.size());
        tl.push_back({r, 0, c, 1, c});
        put(0, r, c, t, 0);
        put(1, r, c, t, 1);
      }
    } else {
      for (size_t k = 0; k < cs.size(); k += 2) {
        const int t = int(tl.size());
        const bool pair = k + 1 < cs.size();
        tl.push_back({r, 0, cs[k], pair ? 0 : -1, pair ? cs[k + 1] : -1});
        put(0, r, cs[k], t, 0);
        if (pair) put(0, r, cs[k + 1], t, 1);
      }
    }
  }
  auto pl = std::make_shared<WidePlan>();
  pl->ntiles = int(tl.size());
  PT_CUDA_CHECK(cudaMalloc(&pl->tiles, tl.size() * sizeof(WideTile)));
  PT_CUDA_CHECK(cudaMemcpy(pl->tiles, tl.data(), tl.size() * sizeof(WideTile), cudaMemcpyHostToDevice));
  PT_CUDA_CHECK(cudaMalloc(&pl->lut, lut.size() * sizeof(int)));
  PT_CUDA_CHECK(cudaMemcpy(pl->lut, lut.data(), lut.size() * sizeof(int), cudaMemcpyHostToDevice));
  ctx->caches[key] = pl;
  return pl;
}

}  // namespace

void gram_tc_wide(pt_ctx* ctx, const c64* A, const c64* B0, c128* C0, const c64* B1, c128* C1, int N1, int N2,
                  size_t ng, double scale, cudaStream_t st, bool herm, bool split3) {
  if (!gram_tc_applies(A, B0, ng) || (B1 && !gram_tc_applies(A, B1, ng)))
    fail(PT_INVALID_ARG, "tensor-core Gram: operands not TMA-addressable");
  herm = herm && (N1 == N2);
  const bool two = B1 != nullptr;
  auto pl = wide_plan(ctx, N1, N2, two, herm);
  const int stages_total = int((2 * ng + WK - 1) / WK);
  // one CTA per SM (~197 KB of shared memory): split K so that one wave fills the GPU
  int splits = std::max(1, ctx->num_sms / pl->ntiles);
  int sps = (stages_total + splits - 1) / splits;
  splits = (stages_total + sps - 1) / sps;
  double* part = static_cast<double*>(
      ctx->get("gram_tc_wide_parts", size_t(splits) * pl->ntiles * 128 * WN * sizeof(double)));
  int* err = static_cast<int*>(ctx->get("gram_tc_err", sizeof(int)));
  if (!ctx->tc_err_clean) {
    PT_CUDA_CHECK(cudaMemsetAsync(err, 0, sizeof(int), st));
    ctx->tc_err_clean = true;
  }
  static DeviceOnce once;
  once([] {
    PT_CUDA_CHECK(cudaFuncSetAttribute(k_gram_tc_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES));
  });
  WideArgs P{reinterpret_cast<const float*>(A),
             reinterpret_cast<const float*>(B0),
             reinterpret_cast<const float*>(two ? B1 : B0),
             N1,
             N2,
             int(2 * ng),
             stages_total,
             sps,
             split3 ? 1 : 0,
             std::max(1, ctx->tc_period)};
  PT_LAUNCH(k_gram_tc_wide, dim3(pl->ntiles, splits), W_THREADS, SMEM_BYTES, st, pl->tiles, P, part, err);
  const size_t n = size_t(N1) * N2;
  const int nbi = (N1 + WB - 1) / WB, nbj = (N2 + WB - 1) / WB;
  PT_LAUNCH_SPLIT_SUM(k_gram_tc_wide_reduce, n, two ? 2u : 1u, splits, st, part, splits, pl->ntiles, pl->lut, nbi, nbj, N1,
                      N2, scale, C0, C1);
}

}  // namespace pt
