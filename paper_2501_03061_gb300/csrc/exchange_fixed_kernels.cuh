// Compile-time pair-FFT exchange kernels (Sec. IV-A1, Eq. vxdiag) on cubic grids with side N.
//
// Four passes per pair batch, all on L2-resident pair fields (one scratch field per pair):
//   plane:      rho = conj(src_i) tgt_j on one z-plane, FFT along x and y;
//   column:     on the (z, x) slab of one y-row: FFT along z, multiply by K(G)/Ng, inverse along z;
//   inv plane:  inverse FFT along y and x of one z-plane, in place (once per pair: with tgt == src
//               the mirrored contribution uses v_ji = conj(v_ij));
//   accumulate: W_t -= sum_c d_c partner_c v_c for every target of the batch (streaming).
// The FFT stages come from fft_fixed.cuh, so all tile index arithmetic is compile-time.
#pragma once

#include <algorithm>

#include "exchange_sched.h"
#include "fft_fixed.cuh"
#include "internal.h"

namespace pt {

namespace {

constexpr int FT = 256;  // threads per CTA of the tile kernels
constexpr int AT = 128;  // threads per CTA of the accumulate kernel
constexpr int AE = 1;    // elements per thread of the accumulate kernel
constexpr int TG = 4;    // targets per CTA of the accumulate kernel
constexpr int CH = 32;   // contributions per target that it holds at a time

template <int N, class T>
constexpr size_t tile_smem() {
  return size_t(N) * kPitch<N> * sizeof(cx<T>) + size_t(N) * sizeof(cx<T>);
}

template <int N, class T>
__global__ void __launch_bounds__(FT) k_fx_fwd_plane(const cx<T>* __restrict__ src, const cx<T>* __restrict__ tgt,
                                                     const double* __restrict__ occ,
                                                     const PairDesc* __restrict__ pairs, cx<T>* __restrict__ scratch,
                                                     const cx<T>* __restrict__ twg) {
  extern __shared__ unsigned char smem_raw[];
  cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* tw = buf + N * kPitch<N>;
  constexpr int PL = N * N;
  constexpr size_t NG = size_t(N) * N * N;
  const int z = blockIdx.x, p = blockIdx.y;
  const PairDesc pd = pairs[p];
  if (pair_skipped(pd, occ)) return;
  for (int t = threadIdx.x; t < N; t += FT) tw[t] = twg[t];
  const cx<T>* a = src + size_t(pd.i) * NG + size_t(z) * PL;
  const cx<T>* b = tgt + size_t(pd.j) * NG + size_t(z) * PL;
#pragma unroll 4
  for (int e = threadIdx.x; e < PL; e += FT) {
    const int y = e / N, x = e - y * N;
    buf[y * kPitch<N> + x] = cmulc(a[e], b[e]);
  }
  __syncthreads();
  cfft_fast<N, false, FT>(buf, tw);  // x
  cfft_slow<N, false, FT>(buf, tw);  // y
  cx<T>* o = scratch + size_t(p) * NG + size_t(z) * PL;
#pragma unroll 4
  for (int e = threadIdx.x; e < PL; e += FT) {
    const int y = e / N, x = e - y * N;
    o[e] = buf[y * kPitch<N> + x];
  }
}

template <int N, class T>
__global__ void __launch_bounds__(FT) k_fx_column(cx<T>* __restrict__ scratch, const T* __restrict__ ktab,
                                                  const double* __restrict__ occ, const PairDesc* __restrict__ pairs,
                                                  const cx<T>* __restrict__ twg) {
  extern __shared__ unsigned char smem_raw[];
  cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* tw = buf + N * kPitch<N>;
  constexpr size_t NG = size_t(N) * N * N;
  const int y = blockIdx.x, p = blockIdx.y;
  const PairDesc pd = pairs[p];
  if (pair_skipped(pd, occ)) return;
  for (int t = threadIdx.x; t < N; t += FT) tw[t] = twg[t];
  cx<T>* f = scratch + size_t(p) * NG;
  // slab tile: row z, column x (z slow, x fast)
#pragma unroll 4
  for (int e = threadIdx.x; e < N * N; e += FT) {
    const int z = e / N, x = e - z * N;
    buf[z * kPitch<N> + x] = f[(size_t(z) * N + y) * N + x];
  }
  __syncthreads();
  cfft_slow<N, false, FT>(buf, tw);  // z
#pragma unroll 4
  for (int e = threadIdx.x; e < N * N; e += FT) {
    const int z = e / N, x = e - z * N;
    buf[z * kPitch<N> + x] = buf[z * kPitch<N> + x] * ktab[(size_t(z) * N + y) * N + x];
  }
  __syncthreads();
  cfft_slow<N, true, FT>(buf, tw);  // inverse z
#pragma unroll 4
  for (int e = threadIdx.x; e < N * N; e += FT) {
    const int z = e / N, x = e - z * N;
    f[(size_t(z) * N + y) * N + x] = buf[z * kPitch<N> + x];
  }
}

template <int N, class T>
__global__ void __launch_bounds__(FT) k_fx_inv_plane(cx<T>* __restrict__ scratch, const double* __restrict__ occ,
                                                     const PairDesc* __restrict__ pairs,
                                                     const cx<T>* __restrict__ twg) {
  extern __shared__ unsigned char smem_raw[];
  cx<T>* buf = reinterpret_cast<cx<T>*>(smem_raw);
  cx<T>* tw = buf + N * kPitch<N>;
  constexpr int PL = N * N;
  constexpr size_t NG = size_t(N) * N * N;
  const int z = blockIdx.x, p = blockIdx.y;
  const PairDesc pd = pairs[p];
  if (pair_skipped(pd, occ)) return;
  for (int t = threadIdx.x; t < N; t += FT) tw[t] = twg[t];
  cx<T>* f = scratch + size_t(p) * NG + size_t(z) * PL;
#pragma unroll 4
  for (int e = threadIdx.x; e < PL; e += FT) {
    const int y = e / N, x = e - y * N;
    buf[y * kPitch<N> + x] = f[e];
  }
  __syncthreads();
  cfft_slow<N, true, FT>(buf, tw);  // inverse y
  cfft_fast<N, true, FT>(buf, tw);  // inverse x
#pragma unroll 4
  for (int e = threadIdx.x; e < PL; e += FT) {
    const int y = e / N, x = e - y * N;
    f[e] = buf[y * kPitch<N> + x];
  }
}

__device__ __forceinline__ float flip_sign(float x, unsigned m) { return __uint_as_float(__float_as_uint(x) ^ m); }
__device__ __forceinline__ double flip_sign(double x, unsigned m) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(m) << 32));
}

__device__ __forceinline__ bool same_bits(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
__device__ __forceinline__ bool same_bits(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

// W_t(r) -= sum_c d_c partner_c(r) v_c(r)  (v conjugated for the mirrored half of a symmetric pair) for TG targets of
// the batch: targets of one tile take their partners in the same order, so d_c partner_c is formed once for them.  In
// FP64 bound by arithmetic (an instruction issues every 64 cycles): six and a half operations per contribution and
// point, signs and the test for d = 0 in integers (eight and a comparison with one target to a CTA).
template <class T>
__global__ void __launch_bounds__(AT) k_fx_accumulate(const cx<T>* __restrict__ scratch, const cx<T>* __restrict__ src,
                                                      const double* __restrict__ occ,
                                                      const TargetDesc* __restrict__ tgts, int nt,
                                                      const Contrib* __restrict__ contribs, cx<T>* __restrict__ out,
                                                      size_t ng) {
  // the contribution lists in shared memory, CH at a time: no chain of dependent loads (list, occupation, field) per
  // contribution
  struct Item {
    int slot, partner;  // slot < 0: no contribution (a skipped pair left its scratch field unwritten)
    unsigned flip;
  };
  __shared__ Item list[TG][CH];
  __shared__ T coef[TG][CH];
  const int t0 = blockIdx.y * TG;
  int most = 0;
#pragma unroll
  for (int u = 0; u < TG; ++u)
    if (t0 + u < nt) most = max(most, tgts[t0 + u].cend - tgts[t0 + u].cbeg);
  const size_t e0 = size_t(blockIdx.x) * (AT * AE) + threadIdx.x;
  cx<T> acc[TG][AE], part[AE];
#pragma unroll
  for (int u = 0; u < TG; ++u)
#pragma unroll
    for (int a = 0; a < AE; ++a) acc[u][a] = czero<T>();
#pragma unroll
  for (int a = 0; a < AE; ++a) part[a] = czero<T>();
  int held = -1;  // the partner in part, with its coefficient
  T held_coef = T(0);
  for (int c0 = 0; c0 < most; c0 += CH) {
    __syncthreads();
    for (int f = threadIdx.x; f < TG * CH; f += AT) {
      const int u = f / CH, c = c0 + f % CH;
      Item it{-1, 0, 0};
      if (t0 + u < nt) {
        const TargetDesc td = tgts[t0 + u];
        if (td.cbeg + c < td.cend) {
          const Contrib cb = contribs[td.cbeg + c];
          const double d = occ[cb.occ];
          if ((__double_as_longlong(d) << 1) != 0) it = Item{cb.slot, cb.partner, cb.conj ? 0x80000000u : 0u};
          coef[u][f % CH] = T(d);
        }
      }
      list[u][f % CH] = it;
    }
    __syncthreads();
    for (int c = 0; c < min(CH, most - c0); ++c) {
      cx<T> w[TG][AE];
#pragma unroll
      for (int u = 0; u < TG; ++u)
#pragma unroll
        for (int a = 0; a < AE; ++a) {
          const size_t e = e0 + size_t(a) * AT;
          w[u][a] = (list[u][c].slot >= 0 && e < ng) ? scratch[size_t(list[u][c].slot) * ng + e] : czero<T>();
        }
#pragma unroll
      for (int u = 0; u < TG; ++u) {
        const Item it = list[u][c];
        if (it.slot < 0) continue;
        const T d = coef[u][c];
        if (it.partner != held || !same_bits(d, held_coef)) {
          held = it.partner;
          held_coef = d;
          const cx<T>* pp = src + size_t(it.partner) * ng;
#pragma unroll
          for (int a = 0; a < AE; ++a)
            if (e0 + size_t(a) * AT < ng) part[a] = pp[e0 + size_t(a) * AT] * d;
        }
#pragma unroll
        for (int a = 0; a < AE; ++a) {
          w[u][a].im = flip_sign(w[u][a].im, it.flip);
          acc[u][a] = acc[u][a] + cmul(part[a], w[u][a]);  // one rounding at the sum's size per contribution
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < TG; ++u) {
    if (t0 + u >= nt) continue;
    const TargetDesc td = tgts[t0 + u];
    cx<T>* o = out + size_t(td.t) * ng;
#pragma unroll
    for (int a = 0; a < AE; ++a) {
      const size_t e = e0 + size_t(a) * AT;
      if (e < ng) o[e] = td.first ? czero<T>() - acc[u][a] : o[e] - acc[u][a];
    }
  }
}

template <int N, class T>
void set_fx_attrs() {
  static DeviceOnce once;
  once([] {
    const int bytes = int(tile_smem<N, T>());
    PT_CUDA_CHECK(
        cudaFuncSetAttribute(k_fx_fwd_plane<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    PT_CUDA_CHECK(cudaFuncSetAttribute(k_fx_column<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    PT_CUDA_CHECK(
        cudaFuncSetAttribute(k_fx_inv_plane<N, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  });
}

// the four passes of one pair batch
template <int N, class T>
void batch_n(const cx<T>* src, const cx<T>* tgt, const double* occ, const PairDesc* pairs, int np,
             const TargetDesc* tgts, int nt, const Contrib* contribs, const T* ktab, const cx<T>* tw, cx<T>* scratch,
             cx<T>* out, cudaStream_t st) {
  set_fx_attrs<N, T>();
  const size_t smem = tile_smem<N, T>();
  constexpr size_t NG = size_t(N) * N * N;
  PT_LAUNCH((k_fx_fwd_plane<N, T>), dim3(N, np), FT, smem, st, src, tgt, occ, pairs, scratch, tw);
  PT_LAUNCH((k_fx_column<N, T>), dim3(N, np), FT, smem, st, scratch, ktab, occ, pairs, tw);
  PT_LAUNCH((k_fx_inv_plane<N, T>), dim3(N, np), FT, smem, st, scratch, occ, pairs, tw);
  const unsigned chunks = unsigned((NG + AT * AE - 1) / (AT * AE));
  PT_LAUNCH(k_fx_accumulate<T>, dim3(chunks, (nt + TG - 1) / TG), AT, 0, st, scratch, src, occ, tgts, nt, contribs, out, NG);
}

}  // namespace

}  // namespace pt
