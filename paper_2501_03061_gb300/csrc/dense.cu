// FP64 dense linear algebra on N x N complex matrices (N up to a few hundred), on the GPU.
//
//   zgemm        C = alpha op(A) op(B) + beta C, op in {N, C (conjugate transpose), T}
//   zgemm_add    C = alpha op(A) op(B) + beta D (D read-only, may differ from C)
//   heev         Hermitian eigen-decomposition by parallel two-sided cyclic Jacobi
//                (round-robin pairing; one launch per round; every 2x2 block of the
//                matrix is updated by J_k^H X J_l in the same launch; entries below the
//                stopping level are not rotated, so late sweeps are mostly copies)
//   cholesky     blocked lower Cholesky (32-wide panels), error flag on a non-positive or
//                non-finite pivot
//   tri_inv      L^{-1} of a lower-triangular matrix, one CTA per column
//   small_solve  m x m (m <= 24) Gaussian elimination with partial pivoting, one thread
// All matrices are row-major complex128: a[i*ld + j].
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace pt {

namespace {

template <class T>
__device__ __forceinline__ cx<T> opval(const cx<T>* A, int lda, char op, int i, int k) {
  // element (i, k) of op(A)
  if (op == 'N') return A[size_t(i) * lda + k];
  cx<T> v = A[size_t(k) * lda + i];
  if (op == 'C') v.im = -v.im;
  return v;
}

constexpr int ZT = 16;

// C = alpha op(A) op(B) + beta D  (D may be C itself, or another matrix with leading dimension ldd)
template <class T>
__global__ void __launch_bounds__(ZT* ZT) k_gemm(char opA, char opB, int m, int n, int k, cx<T> alpha,
                                                 const cx<T>* __restrict__ A, int lda, const cx<T>* __restrict__ B,
                                                 int ldb, cx<T> beta, const cx<T>* D, int ldd, cx<T>* C, int ldc) {
  __shared__ cx<T> As[ZT][ZT + 1];
  __shared__ cx<T> Bs[ZT][ZT + 1];
  const int tx = threadIdx.x % ZT, ty = threadIdx.x / ZT;
  const int i = blockIdx.y * ZT + ty, j = blockIdx.x * ZT + tx;
  cx<T> acc = czero<T>();
  for (int k0 = 0; k0 < k; k0 += ZT) {
    const int ka = k0 + tx, kb = k0 + ty;
    As[ty][tx] = (i < m && ka < k) ? opval(A, lda, opA, i, ka) : czero<T>();
    Bs[ty][tx] = (kb < k && j < n) ? opval(B, ldb, opB, kb, j) : czero<T>();
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < ZT; ++kk) cfma(acc, As[ty][kk], Bs[kk][tx]);
    __syncthreads();
  }
  if (i < m && j < n) {
    cx<T> v = cmul(alpha, acc);
    if (beta.re != T(0) || beta.im != T(0)) v = v + cmul(beta, D[size_t(i) * ldd + j]);
    C[size_t(i) * ldc + j] = v;
  }
}

// The same for small matrices: 8 x 8 tiles with the k range over four groups of threads.  An FP64 instruction issues every 64
// cycles per SM sub-partition, so a 16 x 16 tile of a 48 x 48 product kept 9 of 152 SMs busy for 12 us.
constexpr int ST = 8, SG = 4;
template <class T>
__global__ void __launch_bounds__(ST* ST* SG) k_gemm_small(char opA, char opB, int m, int n, int k, cx<T> alpha,
                                                           const cx<T>* __restrict__ A, int lda, const cx<T>* __restrict__ B,
                                                           int ldb, cx<T> beta, const cx<T>* D, int ldd, cx<T>* C, int ldc) {
  constexpr int KS = 32;  // k per stage
  __shared__ cx<T> As[ST][KS + 1];
  __shared__ cx<T> Bs[KS][ST + 1];
  __shared__ cx<T> red[SG - 1][ST * ST];
  const int t = threadIdx.x, e = t % (ST * ST), g = t / (ST * ST), ty = e / ST, tx = e % ST;
  const int i0 = blockIdx.y * ST, j0 = blockIdx.x * ST, i = i0 + ty, j = j0 + tx;
  cx<T> acc = czero<T>();
  for (int k0 = 0; k0 < k; k0 += KS) {
    for (int f = t; f < ST * KS; f += ST * ST * SG) {
      // consecutive threads on consecutive addresses of op(A) and op(B)
      const int r = opA == 'N' ? f / KS : f % ST, c = opA == 'N' ? f % KS : f / ST;
      As[r][c] = (i0 + r < m && k0 + c < k) ? opval(A, lda, opA, i0 + r, k0 + c) : czero<T>();
      const int q = opB == 'N' ? f / ST : f % KS, l = opB == 'N' ? f % ST : f / KS;
      Bs[q][l] = (k0 + q < k && j0 + l < n) ? opval(B, ldb, opB, k0 + q, j0 + l) : czero<T>();
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KS / SG; ++kk)
      if (k0 + g * (KS / SG) + kk < k) cfma(acc, As[ty][g * (KS / SG) + kk], Bs[g * (KS / SG) + kk][tx]);
    __syncthreads();
  }
  if (g > 0) red[g - 1][e] = acc;
  __syncthreads();
  if (g > 0 || i >= m || j >= n) return;
  for (int q = 0; q < SG - 1; ++q) acc = acc + red[q][e];
  cx<T> v = cmul(alpha, acc);
  if (beta.re != T(0) || beta.im != T(0)) v = v + cmul(beta, D[size_t(i) * ldd + j]);
  C[size_t(i) * ldc + j] = v;
}

// ---------------------------------------------------------------- Jacobi ----
// pair partner of position k in round r of the circle method on Np (even) players
__device__ __forceinline__ void jacobi_pair(int k, int r, int Np, int* p, int* q) {
  auto idx = [&](int i) {  // 1 + (i - 1 + r) mod (Np - 1), r < Np - 1
    const int j = i + r;
    return i == 0 ? 0 : j >= Np ? j - (Np - 1) : j;
  };
  const int a = idx(k), b = idx(Np - 1 - k);
  *p = min(a, b);
  *q = max(a, b);
}

template <class T>
struct Rot {
  T c, s;
  cx<T> u;  // J = [[c, s u], [-s conj(u), c]]
};

__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

// the rotation that annihilates apq (diagonal entries app, aqq), or the identity (s = 0) when |a_pq|^2 <= thr2
// (threshold Jacobi: an entry already below the stopping level is left in place)
template <class T>
__device__ __forceinline__ Rot<T> jacobi_angle(cx<T> apq, T app, T aqq, T thr2) {
  Rot<T> r{T(1), T(0), cx<T>{T(1), T(0)}};
  const T b2 = apq.re * apq.re + apq.im * apq.im;
  if (!(b2 > thr2)) return r;
  // reciprocal square roots in place of square roots and divisions (each a long FP64 sequence on
  // the round's critical path)
  const T rb = rsq(b2);  // 1 / |a_pq|
  const T zeta = (aqq - app) * (T(0.5) * rb);
  const T az = fabs(zeta);
  T t;
  if (az > (sizeof(T) == 8 ? T(1e100) : T(1e15f))) {
    t = T(0.5) / az;  // 1 / (|zeta| + sqrt(1 + zeta^2)) to working precision
  } else {
    const T q2 = T(1) + zeta * zeta;
    t = T(1) / (az + q2 * rsq(q2));
  }
  if (zeta < T(0)) t = -t;
  r.c = rsq(T(1) + t * t);
  r.s = t * r.c;
  r.u = cx<T>{apq.re * rb, apq.im * rb};
  return r;
}
template <class T>
__device__ __forceinline__ Rot<T> jacobi_rot(const cx<T>* A, int N, int p, int q, T thr2) {
  if (q >= N) return Rot<T>{T(1), T(0), cx<T>{T(1), T(0)}};  // padding player
  return jacobi_angle(A[size_t(p) * N + q], A[size_t(p) * N + p].re, A[size_t(q) * N + q].re, thr2);
}

// Z = J_a^H X J_b of a 2 x 2 block; same: the block that the rotation diagonalises
template <class T>
__device__ __forceinline__ void rotate_block(const Rot<T>& a, const Rot<T>& b, bool same, cx<T>& x00, cx<T>& x01,
                                             cx<T>& x10, cx<T>& x11) {
  // Y = J_a^H X:  J^H = [[c, -s u], [s conj(u), c]]
  const cx<T> su = a.u * a.s, suc = conjc(a.u) * a.s;
  const cx<T> y00 = x00 * a.c - cmul(su, x10), y01 = x01 * a.c - cmul(su, x11);
  const cx<T> y10 = cmul(suc, x00) + x10 * a.c, y11 = cmul(suc, x01) + x11 * a.c;
  // Z = Y J_b:  J = [[c, s u], [-s conj(u), c]]
  const cx<T> tu = b.u * b.s, tuc = conjc(b.u) * b.s;
  x00 = y00 * b.c - cmul(y01, tuc);
  x01 = cmul(y00, tu) + y01 * b.c;
  x10 = y10 * b.c - cmul(y11, tuc);
  x11 = cmul(y10, tu) + y11 * b.c;
  if (same) {
    x01 = czero<T>();
    x10 = czero<T>();
    x00.im = T(0);
    x11.im = T(0);
  }
}

constexpr int JB = 8;  // pairs per CTA side (16 x 16 elements): (N/16)^2 CTAs spread over every SM

template <class T>
__global__ void __launch_bounds__(JB* JB) k_jacobi_round(const cx<T>* __restrict__ Ain, cx<T>* __restrict__ Aout,
                                                         cx<T>* __restrict__ V, int N, int Np, int r, T thr2) {
  __shared__ Rot<T> rk[JB], rl[JB];
  __shared__ int pk[JB], qk[JB], pl[JB], ql[JB];
  const int kb = blockIdx.y * JB, lb = blockIdx.x * JB;
  const int half = Np / 2;
  const int t = threadIdx.x;
  pdl_wait();  // the previous round's A and V
  pdl_launch_dependents();
  if (t < JB) {
    const int k = kb + t;
    if (k < half) {
      jacobi_pair(k, r, Np, &pk[t], &qk[t]);
      rk[t] = jacobi_rot(Ain, N, pk[t], qk[t], thr2);
    }
  } else if (t < 2 * JB) {
    const int l = lb + t - JB;
    if (l < half) {
      jacobi_pair(l, r, Np, &pl[t - JB], &ql[t - JB]);
      rl[t - JB] = jacobi_rot(Ain, N, pl[t - JB], ql[t - JB], thr2);
    }
  }
  __syncthreads();
  const int tk = t / JB, tl = t % JB;
  const int k = kb + tk, l = lb + tl;
  if (k < half && l < half) {
    const int p1 = pk[tk], q1 = qk[tk], p2 = pl[tl], q2 = ql[tl];
    const Rot<T> a = rk[tk], b = rl[tl];
    auto get = [&](int i, int j) -> cx<T> {
      return (i < N && j < N) ? Ain[size_t(i) * N + j] : czero<T>();
    };
    const cx<T> x00 = get(p1, p2), x01 = get(p1, q2), x10 = get(q1, p2), x11 = get(q1, q2);
    auto put = [&](int i, int j, cx<T> v) {
      if (i < N && j < N) Aout[size_t(i) * N + j] = v;
    };
    if (a.s == T(0) && b.s == T(0)) {  // both rotations the identity: the block is carried over
      put(p1, p2, x00);
      put(p1, q2, x01);
      put(q1, p2, x10);
      put(q1, q2, x11);
    } else {
      cx<T> z00 = x00, z01 = x01, z10 = x10, z11 = x11;
      rotate_block(a, b, k == l, z00, z01, z10, z11);
      put(p1, p2, z00);
      put(p1, q2, z01);
      put(q1, p2, z10);
      put(q1, q2, z11);
    }
  }
  // V <- V J for the column pairs of this CTA's l-range; the rows are split over the CTAs of the
  // same l-range so every CTA of the grid shares the update
  {
    const int rows_per = (N + gridDim.y - 1) / gridDim.y;
    const int r0 = blockIdx.y * rows_per, r1 = min(N, r0 + rows_per);
    for (int e = t; e < (r1 - r0) * JB; e += JB * JB) {
      const int row = r0 + e / JB, tl2 = e % JB;
      const int l2 = lb + tl2;
      if (l2 >= half) continue;
      const int p2 = pl[tl2], q2 = ql[tl2];
      if (q2 >= N) continue;
      const Rot<T> b = rl[tl2];
      if (b.s == T(0)) continue;  // identity
      const cx<T> vp = V[size_t(row) * N + p2], vq = V[size_t(row) * N + q2];
      const cx<T> tu = b.u * b.s, tuc = conjc(b.u) * b.s;
      V[size_t(row) * N + p2] = vp * b.c - cmul(vq, tuc);
      V[size_t(row) * N + q2] = cmul(vp, tu) + vq * b.c;
    }
  }
}

// ---- FP32 Jacobi on D + E --------------------------------------------------------------------------------------
//
// The off-diagonal part E in FP32, the diagonal D as unevaluated pairs of floats (48 bits), so that differences of
// close eigenvalues are exact: a pass lowers E by FP32's relative precision (~1e-6) however small E already is,
// and finds a basis that is accurate to that times E. Two passes, each made unitary in FP64 and followed by
// X^* A X in FP64, take a matrix from anywhere to 1e-12 of its norm.

// the rotation of (p, q) from E and D; D is updated in place by the owner of the pair
__device__ __forceinline__ Rot<float> jacobi32_angle(c64 apq, float2 dp, float2 dq, float thr2) {
  return jacobi_angle(apq, 0.f, (dq.x - dp.x) + (dq.y - dp.y), thr2);
}
__device__ __forceinline__ float2 pair_add(float2 a, float b) {  // two-sum
  const float s = __fadd_rn(a.x, b), v = __fsub_rn(s, a.x);
  const float e = __fadd_rn(__fadd_rn(__fsub_rn(a.x, __fsub_rn(s, v)), __fsub_rn(b, v)), a.y);
  const float h = __fadd_rn(s, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, s)));
}
__device__ __forceinline__ float2 to_pair(double x) {
  const float h = float(x);
  return make_float2(h, float(x - double(h)));
}
// app -> app - t |apq|, aqq -> aqq + t |apq| with t = s / c
__device__ __forceinline__ void rotate_diag(const Rot<float>& r, c64 apq, float2& dp, float2& dq) {
  if (r.s == 0.f) return;
  const float d = (r.s / r.c) * (apq.re * r.u.re + apq.im * r.u.im);
  dp = pair_add(dp, -d);
  dq = pair_add(dq, d);
}

// when to stop: off and off0 the off-diagonal norms^2 now and at the start, prev after the sweep before
__host__ __device__ inline bool jacobi32_done(double off, double off0, double prev, double floor2, int N) {
  return !(off > floor2) || off <= 1e-14 * N * off0 || (off <= 1e-9 * off0 && off > 0.25 * prev);
}

// One CTA, E and the basis in shared memory (N <= J32_MAX): whole sweeps, two barriers a round (under 1 us at N = 48 against
// 8.7 us of k_jacobi_round, which is a launch and a chain of FP64 instructions).  A thread for each 2 x 2 block of E, as far
// as a CTA has them, and its place in E and V without divisions in the rounds (N = 48, the two passes of a solve:
// 580 -> 445 us).  X: the basis, as FP64; *sweeps_run: the sweeps it took.
constexpr int J32_MAX = 96, J32_THREADS = 1024, J32_SWEEPS = 12;
inline int j32_threads(int N) {
  const int half = (N + 1) / 2;
  return std::min(J32_THREADS, std::max(64, (half * half + 31) / 32 * 32));
}
constexpr size_t j32_smem(int N) { return 2 * size_t(N) * (N | 1) * sizeof(c64); }
__global__ void __launch_bounds__(J32_THREADS) k_jacobi32_cta(const c128* __restrict__ A, int N, float floor2,
                                                              c128* __restrict__ X, double* __restrict__ sweeps_run) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = N | 1, Np = N + (N & 1), half = Np / 2;
  c64* a = reinterpret_cast<c64*>(smem_raw);
  c64* v = a + size_t(N) * P;
  __shared__ Rot<float> rot[J32_MAX / 2];
  __shared__ short2 pq[J32_MAX / 2];
  __shared__ float2 dg[J32_MAX];
  __shared__ float red[J32_THREADS / 32];
  const int t = threadIdx.x, TH = blockDim.x;
  // rows and columns of this thread's first entry, and the step to its next, of a half wide array
  const int first_k = t / half, first_l = t - first_k * half, step_k = TH / half, step_l = TH - step_k * half;
  for (int e = t; e < N * N; e += TH) {
    const int i = e / N, j = e - i * N;
    if (i == j) dg[i] = to_pair(A[e].re);
    a[i * P + j] = to_cx<float>(A[e]);
    v[i * P + j] = c64{i == j ? 1.f : 0.f, 0.f};
  }
  float prev = INFINITY, off0 = 0.f, thr2 = 0.f;
  int sweep = 0;
  for (; sweep < J32_SWEEPS; ++sweep) {
    __syncthreads();
    float off = 0.f;
    for (int e = t; e < N * N; e += TH) {
      const int i = e / N, j = e - i * N;
      const c64 x = a[i * P + j];
      if (i != j) off += x.re * x.re + x.im * x.im;
    }
    for (int o = 16; o; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
    if ((t & 31) == 0) red[t >> 5] = off;
    __syncthreads();
    off = 0.f;
    for (int w = 0; w < TH / 32; ++w) off += red[w];
    if (sweep == 0) {
      off0 = off;
      thr2 = fmaxf(1e-15f * off0, floor2) / (float(N) * float(N));
    }
    // uniform: every thread added the same sums
    if (sweep > 0 && jacobi32_done(off, off0, prev, floor2, N)) break;
    if (sweep > 0) prev = off;
    for (int r = 0; r < Np - 1; ++r) {
      __syncthreads();
      if (t < half) {
        int p, q;
        jacobi_pair(t, r, Np, &p, &q);
        pq[t] = make_short2(short(p), short(q));
        Rot<float> x{1.f, 0.f, c64{1.f, 0.f}};
        if (q < N) {
          const c64 apq = a[p * P + q];
          x = jacobi32_angle(apq, dg[p], dg[q], thr2);
          rotate_diag(x, apq, dg[p], dg[q]);
        }
        rot[t] = x;
      }
      __syncthreads();
      auto next = [&](int& k, int& l) {
        k += step_k, l += step_l;
        if (l >= half) l -= half, ++k;
      };
      for (int k = first_k, l = first_l; k < half; next(k, l)) {
        const Rot<float> x = rot[k], y = rot[l];
        if (x.s == 0.f && y.s == 0.f) continue;
        const int p1 = pq[k].x, q1 = pq[k].y, p2 = pq[l].x, q2 = pq[l].y;
        if (k == l) {
          a[p1 * P + q1] = a[q1 * P + p1] = czero<float>();
          continue;
        }
        const bool in1 = q1 < N, in2 = q2 < N;
        c64 x00 = a[p1 * P + p2], x01 = in2 ? a[p1 * P + q2] : czero<float>();
        c64 x10 = in1 ? a[q1 * P + p2] : czero<float>(), x11 = in1 && in2 ? a[q1 * P + q2] : czero<float>();
        rotate_block(x, y, false, x00, x01, x10, x11);
        a[p1 * P + p2] = x00;
        if (in2) a[p1 * P + q2] = x01;
        if (in1) a[q1 * P + p2] = x10;
        if (in1 && in2) a[q1 * P + q2] = x11;
      }
      for (int row = first_k, l = first_l; row < N; next(row, l)) {
        const Rot<float> y = rot[l];
        const int p = pq[l].x, q = pq[l].y;
        if (y.s == 0.f || q >= N) continue;
        const c64 vp = v[row * P + p], vq = v[row * P + q], tu = y.u * y.s, tuc = conjc(y.u) * y.s;
        v[row * P + p] = vp * y.c - cmul(vq, tuc);
        v[row * P + q] = cmul(vp, tu) + vq * y.c;
      }
    }
  }
  if (t == 0) *sweeps_run = sweep;
  __syncthreads();
  for (int e = t; e < N * N; e += TH) {
    const c64 x = v[(e / N) * P + e % N];
    X[e] = c128{double(x.re), double(x.im)};
  }
}

// The same round over the whole GPU (larger N): E from Ein to Eout, D from Din to Dout, V in place
__global__ void __launch_bounds__(JB* JB) k_jacobi32_round(const c64* __restrict__ Ein, c64* __restrict__ Eout,
                                                           const float2* __restrict__ Din, float2* __restrict__ Dout,
                                                           c64* __restrict__ V, int N, int Np, int r, float thr2) {
  __shared__ Rot<float> rot[2][JB];
  __shared__ int pp[2][JB], qq[2][JB];
  const int kb = blockIdx.y * JB, lb = blockIdx.x * JB, half = Np / 2, t = threadIdx.x;
  pdl_wait();  // the previous round
  pdl_launch_dependents();
  if (t < 2 * JB) {
    const int side = t / JB, i = t % JB, k = (side ? lb : kb) + i;
    if (k < half) {
      int p, q;
      jacobi_pair(k, r, Np, &p, &q);
      pp[side][i] = p;
      qq[side][i] = q;
      Rot<float> x{1.f, 0.f, c64{1.f, 0.f}};
      const bool owner = kb == lb && side == 0;
      if (q < N) {
        const c64 apq = Ein[size_t(p) * N + q];
        float2 dp = Din[p], dq = Din[q];
        x = jacobi32_angle(apq, dp, dq, thr2);
        if (owner) {
          rotate_diag(x, apq, dp, dq);
          Dout[p] = dp;
          Dout[q] = dq;
        }
      } else if (owner) {
        Dout[p] = Din[p];
      }
      rot[side][i] = x;
    }
  }
  __syncthreads();
  const int tk = t / JB, tl = t % JB, k = kb + tk, l = lb + tl;
  if (k < half && l < half) {
    const int p1 = pp[0][tk], q1 = qq[0][tk], p2 = pp[1][tl], q2 = qq[1][tl];
    const Rot<float> x = rot[0][tk], y = rot[1][tl];
    const bool in1 = q1 < N, in2 = q2 < N;
    c64 x00 = Ein[size_t(p1) * N + p2], x01 = in2 ? Ein[size_t(p1) * N + q2] : czero<float>();
    c64 x10 = in1 ? Ein[size_t(q1) * N + p2] : czero<float>(), x11 = in1 && in2 ? Ein[size_t(q1) * N + q2] : czero<float>();
    if (x.s != 0.f || y.s != 0.f) {
      if (k == l) x01 = x10 = czero<float>();
      else rotate_block(x, y, false, x00, x01, x10, x11);
    }
    Eout[size_t(p1) * N + p2] = x00;
    if (in2) Eout[size_t(p1) * N + q2] = x01;
    if (in1) Eout[size_t(q1) * N + p2] = x10;
    if (in1 && in2) Eout[size_t(q1) * N + q2] = x11;
  }
  // V <- V J for this CTA's l range, the rows split over the CTAs of that range
  const int rows = (N + gridDim.y - 1) / gridDim.y, r0 = blockIdx.y * rows, r1 = min(N, r0 + rows);
  for (int e = t; e < (r1 - r0) * JB; e += JB * JB) {
    const int row = r0 + e / JB, i = e % JB;
    if (lb + i >= half || qq[1][i] >= N || rot[1][i].s == 0.f) continue;
    const Rot<float> y = rot[1][i];
    c64 *vp = V + size_t(row) * N + pp[1][i], *vq = V + size_t(row) * N + qq[1][i];
    const c64 a = *vp, b = *vq, tu = y.u * y.s, tuc = conjc(y.u) * y.s;
    *vp = a * y.c - cmul(b, tuc);
    *vq = cmul(a, tu) + b * y.c;
  }
}

__global__ void __launch_bounds__(256) k_jacobi32_start(const c128* __restrict__ A, int N, c64* __restrict__ E,
                                                        float2* __restrict__ D, c64* __restrict__ V) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= N * N) return;
  const int i = e / N, j = e - i * N;
  E[e] = i == j ? czero<float>() : to_cx<float>(A[e]);
  if (i == j) D[i] = to_pair(A[e].re);
  V[e] = c64{i == j ? 1.f : 0.f, 0.f};
}
__global__ void __launch_bounds__(256) k_widen(const c64* __restrict__ V32, int n, c128* __restrict__ X) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e < n) X[e] = c128{double(V32[e].re), double(V32[e].im)};
}

// A = (S + S^*)/2 and V = V0 (identity when V0 is NULL)
__global__ void k_herm_part_and_basis(const c128* __restrict__ S, c128* __restrict__ A, const c128* __restrict__ V0,
                                      c128* __restrict__ V, int N) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int i = e / N, j = e % N;
  const c128 a = S[size_t(i) * N + j], b = S[size_t(j) * N + i];
  A[e] = c128{0.5 * (a.re + b.re), 0.5 * (a.im - b.im)};
  V[e] = V0 ? V0[e] : c128{i == j ? 1.0 : 0.0, 0.0};
}

// sums of |offdiag|^2 and |all|^2: one partial pair per block (OFF_BLOCKS blocks), then one thread
// adds the partials in order
constexpr int OFF_BLOCKS = 64;
template <class T>
__global__ void __launch_bounds__(256) k_offnorm_part(const cx<T>* __restrict__ A, int N, double* __restrict__ part) {
  pdl_wait();  // the last Jacobi round
  double off = 0, all = 0;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < N * N; e += OFF_BLOCKS * 256) {
    const double v = double(A[e].re) * double(A[e].re) + double(A[e].im) * double(A[e].im);
    all += v;
    if (e / N != e % N) off += v;
  }
  __shared__ double so[8], sa[8];
  for (int o = 16; o; o >>= 1) {
    off += __shfl_down_sync(0xffffffffu, off, o);
    all += __shfl_down_sync(0xffffffffu, all, o);
  }
  if ((threadIdx.x & 31) == 0) {
    so[threadIdx.x >> 5] = off;
    sa[threadIdx.x >> 5] = all;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int w = 0; w < 8; ++w) {
      a += so[w];
      b += sa[w];
    }
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
  }
}
__global__ void k_offnorm_sum(const double* __restrict__ part, double* __restrict__ out) {
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int k = 0; k < OFF_BLOCKS; ++k) {
      a += part[2 * k];
      b += part[2 * k + 1];
    }
    out[0] = a;
    out[1] = b;
  }
}

// ascending sort of the diagonal with the matching columns of V: a rank sort on order-preserving
// integer keys of the doubles (an FP64 comparison issues at the FP64 rate here), then the column
// permutation over the whole grid
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__global__ void k_eig_keys(const c128* __restrict__ A, int N, unsigned long long* __restrict__ key) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) key[i] = order_key(A[size_t(i) * N + i].re);
}
__global__ void k_eig_rank(const c128* __restrict__ A, const unsigned long long* __restrict__ key, int N,
                           int* __restrict__ rank, double* __restrict__ d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const unsigned long long ki = key[i];
  int r = 0;
  for (int j = 0; j < N; ++j) {
    const unsigned long long kj = key[j];  // the same j across the warp: one broadcast load
    r += (kj < ki) || (kj == ki && j < i);
  }
  rank[i] = r;
  d[r] = A[size_t(i) * N + i].re;
}
__global__ void k_eig_permute(const c128* __restrict__ V, const int* __restrict__ rank, int N, c128* __restrict__ Q) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int row = e / N, i = e - row * N;
  Q[size_t(row) * N + rank[i]] = V[e];
}

// ---------------------------------------------------------------- Cholesky ----
// Right-looking blocked Cholesky with CB-wide panels.  Per panel: the diagonal block is
// factored (and inverted) in one CTA's shared memory, the panel below is solved against the
// inverse of the diagonal block, and the trailing lower triangle gets a rank-CB update.
constexpr int CB = 32;

// a positive finite number, tested on its bits (an FP64 comparison issues at the FP64 rate here)
__device__ __forceinline__ bool good_pivot(float x) {
  const int b = __float_as_int(x);
  return b > 0 && b < 0x7f800000;
}
__device__ __forceinline__ bool good_pivot(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool is_zero_bits(float x) { return __float_as_int(x) == 0; }
__device__ __forceinline__ bool is_zero_bits(double x) { return __double_as_longlong(x) == 0; }

// Factor and inverse of a diagonal block as A = U D U^* (U unit lower triangular): step k subtracts column k's outer product
// from the trailing triangle and column k from the rows of U^{-1} below it; L = U D^{1/2} and L^{-1} = D^{-1/2} U^{-1}
// at the end.  A step is one barrier: warp 0 updates the next pivot and forms its reciprocal while the other
// warps do the rest, so the FP64 chain (six dependent operations and a reciprocal) and the FP64 work run side by
// side.  (With a square root, the column and the update behind barriers of their own and the inverse row by row after
// them a 32 x 32 FP64 block took 95 us; this takes 52.)
template <class T>
__global__ void __launch_bounds__(256) k_chol_diag(cx<T>* __restrict__ A, int N, int kb, int bs,
                                                   cx<T>* __restrict__ Winv, int* __restrict__ info) {
  __shared__ cx<T> a[CB][CB + 1];
  __shared__ cx<T> x[CB][CB + 1];
  // lower triangle (i >= j) listed column by column: entry (j, i) at j*bs - j(j-1)/2 + (i - j), so
  // the trailing triangle of step k (j > k) is one contiguous range, its first entry the next pivot
  __shared__ unsigned short tri[CB * (CB + 1) / 2];
  // reciprocals of the pivots (zero: the pivot is not positive and finite) and of their square roots
  __shared__ T rd[CB], rs[CB];
  pdl_wait();  // the previous panel's trailing update
  pdl_launch_dependents();
  if (*info) return;
  const int tid = threadIdx.x;
  for (int e = tid; e < bs * bs; e += blockDim.x) {
    const int i = e / bs, j = e % bs;
    a[i][j] = A[size_t(kb + i) * N + kb + j];
    x[i][j] = cx<T>{T(i == j ? 1 : 0), T(0)};
    if (i >= j) tri[j * bs - j * (j - 1) / 2 + (i - j)] = static_cast<unsigned short>((j << 8) | i);
  }
  __syncthreads();
  auto pivot = [&](int k) {  // one thread: a[k][k] is final
    const T d = a[k][k].re;
    rd[k] = good_pivot(d) ? T(1) / d : T(0);
  };
  if (tid == 0) pivot(0);
  __syncthreads();
  const int tri_end = bs * (bs + 1) / 2;
  for (int k = 0; k < bs; ++k) {
    const T r = rd[k];
    if (is_zero_bits(r)) {  // uniform: written before the barrier behind this step, which writes rd[k + 1] alone
      if (tid == 0) *info = kb + k + 1;
      return;
    }
    const int first = (k + 1) * bs - (k + 1) * k / 2;
    if (tid < 32) {
      if (tid == 0 && k + 1 < bs) {
        const cx<T> c = a[k + 1][k];
        a[k + 1][k + 1].re -= c.re * (c.re * r) + c.im * (c.im * r);  // c squared would leave the range first
        pivot(k + 1);
      }
    } else {
      const int n1 = max(0, tri_end - first - 1), n2 = (bs - 1 - k) * (k + 1);
      for (int e = tid - 32; e < n1 + n2; e += 256 - 32) {
        if (e < n1) {
          const int i = tri[first + 1 + e] & 255, j = tri[first + 1 + e] >> 8;
          a[i][j] = a[i][j] - cmulc(a[j][k] * r, a[i][k]);
        } else {
          const int f = e - n1, i = k + 1 + f / (k + 1), j = f % (k + 1);
          x[i][j] = x[i][j] - cmul(a[i][k] * r, x[k][j]);
        }
      }
    }
    __syncthreads();
  }
  if (tid < bs) rs[tid] = rsq(a[tid][tid].re);
  __syncthreads();
  for (int e = tid; e < bs * bs; e += blockDim.x) {
    const int i = e / bs, j = e % bs;
    if (j <= i) A[size_t(kb + i) * N + kb + j] = j == i ? cx<T>{a[i][i].re * rs[i], T(0)} : a[i][j] * rs[j];
    Winv[i * CB + j] = j <= i ? x[i][j] * rs[i] : czero<T>();
  }
}

// L_ik = A_ik L_kk^{-*} for the rows below the diagonal block (8 rows per CTA)
template <class T>
__global__ void __launch_bounds__(256) k_chol_panel(cx<T>* __restrict__ A, int N, int kb, int bs,
                                                    const cx<T>* __restrict__ Winv, const int* __restrict__ info) {
  __shared__ cx<T> w[CB][CB + 1];
  __shared__ cx<T> r[8][CB + 1];
  pdl_wait();  // the diagonal block and its inverse
  pdl_launch_dependents();
  if (*info) return;
  const int tid = threadIdx.x;
  const int i0 = kb + bs + blockIdx.x * 8;
  for (int e = tid; e < bs * bs; e += blockDim.x) w[e / bs][e % bs] = Winv[(e / bs) * CB + (e % bs)];
  for (int e = tid; e < 8 * bs; e += blockDim.x) {
    const int ii = e / bs, p = e % bs;
    r[ii][p] = (i0 + ii < N) ? A[size_t(i0 + ii) * N + kb + p] : czero<T>();
  }
  __syncthreads();
  const int ii = tid / CB, j = tid % CB;
  if (i0 + ii < N && j < bs) {
    cx<T> acc = czero<T>();
    // (L_kk^{-*})[p][j] = conj(Winv[j][p]), nonzero for p <= j
    for (int p = 0; p <= j; ++p) acc = acc + cmul(r[ii][p], conjc(w[j][p]));
    A[size_t(i0 + ii) * N + kb + j] = acc;
  }
}

// trailing update A[i][j] -= sum_p L[i][kb+p] conj(L[j][kb+p]) for kb+bs <= j <= i < N
template <class T>
__global__ void __launch_bounds__(256) k_chol_update(cx<T>* __restrict__ A, int N, int kb, int bs,
                                                     const int* __restrict__ info) {
  pdl_wait();  // the panel below the diagonal block
  pdl_launch_dependents();
  if (*info) return;
  const int t0 = kb + bs;
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj > bi) return;
  __shared__ cx<T> li[16][CB + 1], lj[16][CB + 1];
  const int tid = threadIdx.x;
  const int ib = t0 + bi * 16, jb = t0 + bj * 16;
  for (int e = tid; e < 16 * bs; e += blockDim.x) {
    const int q = e / bs, p = e % bs;
    li[q][p] = (ib + q < N) ? A[size_t(ib + q) * N + kb + p] : czero<T>();
    lj[q][p] = (jb + q < N) ? A[size_t(jb + q) * N + kb + p] : czero<T>();
  }
  __syncthreads();
  const int i = ib + tid / 16, j = jb + tid % 16;
  if (i < N && j < N && j <= i) {
    cx<T> acc = czero<T>();
    for (int p = 0; p < bs; ++p) acc = acc + cmulc(lj[tid % 16][p], li[tid / 16][p]);
    A[size_t(i) * N + j] = A[size_t(i) * N + j] - acc;
  }
}

template <class T>
__global__ void k_chol_finish(const cx<T>* __restrict__ A, int N, cx<T>* __restrict__ L, const int* __restrict__ info) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N || *info) return;
  const int i = e / N, j = e % N;
  L[e] = (j > i) ? czero<T>() : A[e];
}

// out = U diag(f(lam)) (scale columns), f = lam^power
__global__ void k_scale_cols_pow(const c128* __restrict__ U, const double* __restrict__ lam, int N, double power,
                                 c128* __restrict__ out, int* __restrict__ info) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int j = e % N;
  const double l = lam[j];
  if (!(l > 0.0)) {
    *info = 1;
    out[e] = czero<double>();
    return;
  }
  out[e] = U[e] * pow(l, power);
}

__global__ void k_small_solve(const double* __restrict__ G, const double* __restrict__ rhs, int m, double reg,
                              double* __restrict__ x) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a[24][25];
  double tr = 0;
  for (int i = 0; i < m; ++i) tr += G[i * m + i];
  const double shift = reg * (tr > 0 ? tr / m : 1.0);
  for (int i = 0; i < m; ++i) {
    for (int j = 0; j < m; ++j) a[i][j] = G[i * m + j] + (i == j ? shift : 0.0);
    a[i][m] = rhs[i];
  }
  for (int c = 0; c < m; ++c) {
    int piv = c;
    for (int r = c + 1; r < m; ++r)
      if (fabs(a[r][c]) > fabs(a[piv][c])) piv = r;
    if (piv != c)
      for (int j = c; j <= m; ++j) {
        const double t = a[c][j];
        a[c][j] = a[piv][j];
        a[piv][j] = t;
      }
    const double d = a[c][c];
    if (d == 0.0) continue;
    for (int r = c + 1; r < m; ++r) {
      const double f = a[r][c] / d;
      for (int j = c; j <= m; ++j) a[r][j] -= f * a[c][j];
    }
  }
  for (int c = m - 1; c >= 0; --c) {
    double s = a[c][m];
    for (int j = c + 1; j < m; ++j) s -= a[c][j] * x[j];
    x[c] = (a[c][c] != 0.0) ? s / a[c][c] : 0.0;
  }
}

}  // namespace

// ------------------------------------------------------------------------------------------
template <class T>
void gemm(char opA, char opB, int m, int n, int k, cx<T> alpha, const cx<T>* A, int lda, const cx<T>* B, int ldb,
          cx<T> beta, const cx<T>* D, int ldd, cx<T>* C, int ldc, cudaStream_t st) {
  // small tiles while 16 x 16 ones would leave SMs idle (152 of them): FP64 N = 48 17.6 -> 9 us a product, N = 75 23 -> 9
  if (((n + ZT - 1) / ZT) * ((m + ZT - 1) / ZT) < 152) {
    PT_LAUNCH(k_gemm_small<T>, dim3((n + ST - 1) / ST, (m + ST - 1) / ST), ST * ST * SG, 0, st, opA, opB, m, n, k, alpha, A,
              lda, B, ldb, beta, D, ldd, C, ldc);
    return;
  }
  dim3 grid((n + ZT - 1) / ZT, (m + ZT - 1) / ZT);
  PT_LAUNCH(k_gemm<T>, grid, ZT * ZT, 0, st, opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, D, ldd, C, ldc);
}
template void gemm<float>(char, char, int, int, int, c64, const c64*, int, const c64*, int, c64, const c64*, int, c64*,
                          int, cudaStream_t);
template void gemm<double>(char, char, int, int, int, c128, const c128*, int, const c128*, int, c128, const c128*, int,
                           c128*, int, cudaStream_t);

void zgemm(char opA, char opB, int m, int n, int k, c128 alpha, const c128* A, int lda, const c128* B, int ldb,
           c128 beta, c128* C, int ldc, cudaStream_t st) {
  gemm<double>(opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, C, ldc, st);
}

void zgemm_add(char opA, char opB, int m, int n, int k, c128 alpha, const c128* A, int lda, const c128* B, int ldb,
               c128 beta, const c128* D, int ldd, c128* C, int ldc, cudaStream_t st) {
  gemm<double>(opA, opB, m, n, k, alpha, A, lda, B, ldb, beta, D, ldd, C, ldc, st);
}

int heev(pt_ctx* ctx, const c128* S, int N, c128* Q, double* d, cudaStream_t st, int max_sweeps, const c128* Q0,
         double rel_tol) {
  const int Np = N + (N & 1);
  c128* A0 = static_cast<c128*>(ctx->get("heev_A0", size_t(N) * N * sizeof(c128)));
  c128* A1 = static_cast<c128*>(ctx->get("heev_A1", size_t(N) * N * sizeof(c128)));
  c128* V = static_cast<c128*>(ctx->get("heev_V", size_t(N) * N * sizeof(c128)));
  // the norms, the sweeps of a pass in one CTA, the blocks' sums
  double* nrm = static_cast<double*>(ctx->get("heev_norm", (2 * OFF_BLOCKS + 3) * sizeof(double)));
  if (Q0) {
    // warm start: rotate into the basis Q0 (Jacobi then starts from a nearly diagonal matrix when
    // Q0 diagonalises a nearby matrix) and accumulate the rotations onto Q0
    zgemm('N', 'N', N, N, N, c128{1, 0}, S, N, Q0, N, c128{0, 0}, A1, N, st);
    zgemm('C', 'N', N, N, N, c128{1, 0}, Q0, N, A1, N, c128{0, 0}, V, N, st);
    PT_LAUNCH(k_herm_part_and_basis, (N * N + 255) / 256, 256, 0, st, V, A0, Q0, A1, N);
    std::swap(V, A1);
  } else {
    PT_LAUNCH(k_herm_part_and_basis, (N * N + 255) / 256, 256, 0, st, S, A0, nullptr, V, N);
  }
  const int half = Np / 2;
  dim3 grid((half + JB - 1) / JB, (half + JB - 1) / JB);
  double h[3] = {0, 0, 0};
  int sweeps = 0;            // of all passes
  bool cta_pass = false;     // h[2] will hold a pass's sweeps
  auto norms = [&](auto* A) {
    PT_LAUNCH_PDL((k_offnorm_part<std::decay_t<decltype(A->re)>>), OFF_BLOCKS, 256, 0, st, A, N, nrm + 3);
    PT_LAUNCH(k_offnorm_sum, 1, 32, 0, st, nrm + 3, nrm);
    PT_CUDA_CHECK(cudaMemcpyAsync(h, nrm, sizeof(h), cudaMemcpyDeviceToHost, st));
    PT_CUDA_CHECK(cudaStreamSynchronize(st));
    if (cta_pass) sweeps += int(h[2]);
    cta_pass = false;
    if (!std::isfinite(h[1])) fail(PT_NONFINITE, "non-finite entry in the matrix to diagonalise");
  };
  // Where the caller asks for less than FP64 rounding (rel_tol): FP32 passes on D + E (see k_jacobi32_cta), each basis
  // made unitary in FP64 by two Newton-Schulz steps (X <- X (3 I - X^* X)/2, the error squared each time) and
  // A <- X^* A X in FP64.  Two passes usually meet the tolerance, whose test stays that of the FP64 sweeps below, which
  // finish the rest.  A pass costs seven FP64 products and its sweeps (N = 48: 2.05 -> about 0.67 ms a solve; N = 320, a launch
  // per FP32 round: 25 -> 15 ms).
  for (int pass = 0; rel_tol > 0.0 && pass < 3; ++pass) {
    const double before = h[0];
    norms(A0);
    const double floor2 = 0.01 * rel_tol * rel_tol * h[1];
    if (!(h[1] > 1e-6 && h[1] < 1e12) || h[0] <= rel_tol * rel_tol * h[1]) break;
    if (pass > 0 && h[0] > 1e-4 * before) break;  // no longer gaining: leave it to the FP64 sweeps
    c128* X0 = static_cast<c128*>(ctx->get("heev_X0", size_t(N) * N * sizeof(c128)));
    c128* X1 = static_cast<c128*>(ctx->get("heev_X1", size_t(N) * N * sizeof(c128)));
    c128* G = static_cast<c128*>(ctx->get("heev_G", size_t(N) * N * sizeof(c128)));
    const int nb = (N * N + 255) / 256;
    if (N <= J32_MAX) {
      static DeviceOnce once;
      once([] {
        PT_CUDA_CHECK(
            cudaFuncSetAttribute(k_jacobi32_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, int(j32_smem(J32_MAX))));
      });
      PT_LAUNCH(k_jacobi32_cta, 1, j32_threads(N), j32_smem(N), st, A0, N, float(floor2), X0, nrm + 2);
      cta_pass = true;
    } else {
      // E and V in buffers that are free until the products below
      c64 *e0 = reinterpret_cast<c64*>(G), *e1 = e0 + size_t(N) * N, *v32 = reinterpret_cast<c64*>(X1);
      float2* d0 = static_cast<float2*>(ctx->get("heev_D32", 2 * size_t(N) * sizeof(float2)));
      float2* d1 = d0 + N;
      PT_LAUNCH(k_jacobi32_start, nb, 256, 0, st, A0, N, e0, d0, v32);
      const double off0 = h[0];
      const float thr2 = float(std::max(1e-15 * off0, floor2) / (double(N) * double(N)));
      double prev = INFINITY;
      for (int sweep = 0; sweep < J32_SWEEPS; ++sweep) {
        if (sweep > 0) {
          norms(e0);
          if (jacobi32_done(h[0], off0, prev, floor2, N)) break;
          prev = h[0];
        }
        for (int r = 0; r < Np - 1; ++r) {
          PT_LAUNCH_PDL(k_jacobi32_round, grid, JB * JB, 0, st, e0, e1, d0, d1, v32, N, Np, r, thr2);
          std::swap(e0, e1);
          std::swap(d0, d1);
        }
        ++sweeps;
      }
      h[0] = off0;
      PT_LAUNCH(k_widen, nb, 256, 0, st, v32, N * N, X0);
    }
    const c128 one{1, 0}, zero{0, 0};
    for (int it = 0; it < 2; ++it) {
      zgemm('C', 'N', N, N, N, one, X0, N, X0, N, zero, G, N, st);
      zgemm_add('N', 'N', N, N, N, c128{-0.5, 0}, X0, N, G, N, c128{1.5, 0}, X0, N, X1, N, st);
      std::swap(X0, X1);
    }
    zgemm('N', 'N', N, N, N, one, A0, N, X0, N, zero, G, N, st);
    zgemm('C', 'N', N, N, N, one, X0, N, G, N, zero, A1, N, st);
    zgemm('N', 'N', N, N, N, one, V, N, X0, N, zero, G, N, st);
    PT_LAUNCH(k_herm_part_and_basis, nb, 256, 0, st, A1, A0, G, V, N);
  }
  double prev_off = INFINITY;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    norms(A0);
    // Converged when the off-diagonal norm is at the FP64 rounding floor (eps * sqrt(N) * ||A||),
    // or when, already small, a sweep no longer reduces it (cyclic Jacobi converges
    // quadratically, so a stalled sweep means rounding noise).
    const double floor2 = 1e-32 * double(N) * h[1];
    if (h[0] <= floor2 || h[0] == 0.0) break;
    if (h[0] <= rel_tol * rel_tol * h[1]) break;
    if (h[0] <= 1e-24 * h[1] && h[0] > 0.25 * prev_off) break;
    prev_off = h[0];
    // entries with |a_pq|^2 at or below the stopping level spread over all N^2 entries are not
    // rotated: all of them together stay within the stopping test, and late sweeps, where most
    // entries are there, skip their FP64 arithmetic
    const double stop2 = rel_tol > 0.0 ? rel_tol * rel_tol * h[1] : floor2;
    const double thr2 = std::max(1e-280, stop2 / (double(N) * double(N)));
    for (int r = 0; r < Np - 1; ++r) {
      PT_LAUNCH_PDL(k_jacobi_round<double>, grid, JB * JB, 0, st, A0, A1, V, N, Np, r, thr2);
      std::swap(A0, A1);
    }
    ++sweeps;
  }
  auto* key = static_cast<unsigned long long*>(ctx->get("heev_key", size_t(N) * sizeof(unsigned long long)));
  int* rank = static_cast<int*>(ctx->get("heev_rank", size_t(N) * sizeof(int)));
  PT_LAUNCH(k_eig_keys, (N + 255) / 256, 256, 0, st, A0, N, key);
  PT_LAUNCH(k_eig_rank, (N + 127) / 128, 128, 0, st, A0, key, N, rank, d);
  PT_LAUNCH(k_eig_permute, (N * N + 255) / 256, 256, 0, st, V, rank, N, Q);
  return sweeps;
}

template <class T>
void cholesky(pt_ctx* ctx, cx<T>* A, int N, cx<T>* L, int* info, cudaStream_t st) {
  // the inverses of all diagonal blocks are kept (rows kb..kb+bs of an N x CB array) for tri_inv_lower
  cx<T>* winv_all = static_cast<cx<T>*>(
      ctx->get(sizeof(T) == 8 ? "chol_winv_all" : "chol_winv_all32", size_t(N) * CB * sizeof(cx<T>)));
  PT_CUDA_CHECK(cudaMemsetAsync(info, 0, sizeof(int), st));
  for (int kb = 0; kb < N; kb += CB) {
    const int bs = std::min(CB, N - kb);
    cx<T>* winv = winv_all + size_t(kb) * CB;
    PT_LAUNCH_PDL(k_chol_diag<T>, 1, 256, 0, st, A, N, kb, bs, winv, info);
    const int rest = N - kb - bs;
    if (rest <= 0) break;
    PT_LAUNCH_PDL(k_chol_panel<T>, (rest + 7) / 8, 256, 0, st, A, N, kb, bs, winv, info);
    const int nt = (rest + 15) / 16;
    PT_LAUNCH_PDL(k_chol_update<T>, dim3(nt, nt), 256, 0, st, A, N, kb, bs, info);
  }
  PT_LAUNCH(k_chol_finish<T>, (N * N + 255) / 256, 256, 0, st, A, N, L, info);
}
template void cholesky<float>(pt_ctx*, c64*, int, c64*, int*, cudaStream_t);
template void cholesky<double>(pt_ctx*, c128*, int, c128*, int*, cudaStream_t);

// X = 0 except the diagonal CB-blocks, which take the inverses cholesky() kept
template <class T>
__global__ void k_tri_inv_leaves(const cx<T>* __restrict__ winv_all, int N, cx<T>* __restrict__ X) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * N) return;
  const int i = e / N, j = e % N;
  const int bi = i / CB, bj = j / CB;
  X[e] = (bi == bj) ? winv_all[size_t(i) * CB + (j - bj * CB)] : czero<T>();
}

template <class T>
void tri_inv_lower(pt_ctx* ctx, const cx<T>* L, int N, cx<T>* X, cudaStream_t st) {
  // Bottom-up block inversion: for [L11 0; L21 L22] with X11 = L11^{-1}, X22 = L22^{-1} known,
  // X21 = -X22 (L21 X11).  Leaves are the CB x CB inverses from the preceding cholesky().
  const cx<T>* winv_all = static_cast<const cx<T>*>(
      ctx->get(sizeof(T) == 8 ? "chol_winv_all" : "chol_winv_all32", size_t(N) * CB * sizeof(cx<T>)));
  cx<T>* Tm = static_cast<cx<T>*>(ctx->get(sizeof(T) == 8 ? "tri_inv_T" : "tri_inv_T32", size_t(N) * N * sizeof(cx<T>)));
  PT_LAUNCH(k_tri_inv_leaves<T>, (N * N + 255) / 256, 256, 0, st, winv_all, N, X);
  const cx<T> one{T(1), T(0)}, mone{T(-1), T(0)}, zero{T(0), T(0)};
  for (int s = CB; s < N; s *= 2) {
    for (int i0 = 0; i0 + s < N; i0 += 2 * s) {
      const int n1 = s, n2 = std::min(s, N - i0 - s);
      const cx<T>* X11 = X + size_t(i0) * N + i0;
      const cx<T>* X22 = X + size_t(i0 + s) * N + (i0 + s);
      const cx<T>* L21 = L + size_t(i0 + s) * N + i0;
      cx<T>* X21 = X + size_t(i0 + s) * N + i0;
      gemm<T>('N', 'N', n2, n1, n1, one, L21, N, X11, N, zero, Tm, n1, Tm, n1, st);
      gemm<T>('N', 'N', n2, n1, n2, mone, X22, N, Tm, n1, zero, X21, N, X21, N, st);
    }
  }
}
template void tri_inv_lower<float>(pt_ctx*, const c64*, int, c64*, cudaStream_t);
template void tri_inv_lower<double>(pt_ctx*, const c128*, int, c128*, cudaStream_t);

void scale_cols_pow(const c128* U, const double* lam, int N, double power, c128* out, int* info, cudaStream_t st) {
  PT_LAUNCH(k_scale_cols_pow, (N * N + 255) / 256, 256, 0, st, U, lam, N, power, out, info);
}

__global__ void k_set_identity(c128* __restrict__ A, int N) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < N * N) A[e] = c128{(e / N == e % N) ? 1.0 : 0.0, 0.0};
}

__global__ void k_add_diagonal(c128* __restrict__ A, int N, double v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) A[size_t(i) * N + i].re += v;
}

void set_identity(c128* A, int N, cudaStream_t st) {
  PT_LAUNCH(k_set_identity, (N * N + 255) / 256, 256, 0, st, A, N);
}

void add_diagonal(c128* A, int N, double v, cudaStream_t st) {
  PT_LAUNCH(k_add_diagonal, (N + 255) / 256, 256, 0, st, A, N, v);
}

void small_solve(const double* G, const double* rhs, int m, double reg, double* x, cudaStream_t st) {
  if (m > 24) fail(PT_INVALID_ARG, "small_solve supports m <= 24");
  PT_LAUNCH(k_small_solve, 1, 32, 0, st, G, rhs, m, reg, x);
}

}  // namespace pt
