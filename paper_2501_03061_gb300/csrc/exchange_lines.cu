// FP32 pair-FFT exchange with whole lines in registers: cubic grids (the sides of PT_FIXED_SIZES) here, the others
// in exchange_lines_axes.cu
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
// and the passes run at 25-45% of the issue rate, 35-60% of the L1 rate and, at 64^3, 4.2-5.2 TB/s of memory
// (0.63-0.78 of a copy), waiting on the loads
// and stores of lines between the transforms.  Measured on GB300, one V_x application, all pairs
// symmetric (this form against the tile kernels, at 64 against the TMA pipeline it replaced):
//   24^3 N = 64   0.22 against 0.67 ms      48^3 N = 128   6.7 against 18.0 ms
//   36^3 N = 96   1.69 against 4.66 ms      64^3 N = 96    9.7 against 14.4 ms, N = 320 105.5 against 157.4
// i.e. 0.007-0.009 ns per pair and grid point against 0.012 (64^3) and 0.020-0.026.
#include "exchange_lines.cuh"
#include "fft_fixed.cuh"

namespace pt {

namespace {

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
  const int regs = N <= 24 ? 80 : N == 30 ? 128 : N <= 32 ? 96 : N <= 40 ? 128 : 168;
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

template <int N>
void run_tile(const Tile& t, const c64* src, const c64* tgt, const double* occ, const float* kt, c64* scratch, c64* out,
              int sms, cudaStream_t st) {
  static DeviceOnce once;
  once([] {
    PT_CUDA_CHECK(cudaFuncSetAttribute(k_xl_plane<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kPlaneSmem<N>)));
  });
  run_zfwd<N, N * N>(t, src, tgt, occ, scratch, N * N, st);
  PT_LAUNCH(k_xl_plane<N>, dim3(N / planes(N), t.nj, t.ni), kPlaneThreads<N>, kPlaneSmem<N>, st, t, occ, kt, scratch);
  run_accum<N, N * N>(t, src, occ, scratch, out, N * N, sms, st);
}

}  // namespace

bool exchange_lines_applies(const pt_ctx* ctx, const pt_grid& g) {
  const bool lines = fixed_cubic(g) || (line_length(g.nx) && line_length(g.ny) && line_length(g.nz));
  return lines && (exchange64_applies(g) ? ctx->exchange64_engine == 0 : ctx->exchange64_engine != 1);
}

long long exchange_lines(pt_ctx* ctx, const c64* src, const double* occ, int N, const c64* tgt, int M, bool sym, c64* out,
                         const pt_grid& g, const pt_kernel& k, size_t budget, cudaStream_t st) {
  const size_t field = ng_of(g) * sizeof(c64);
  int B = int(std::floor(std::sqrt(double(std::max<size_t>(1, budget / field)))));
  B = std::max(1, std::min({B, std::max(N, M), MAXB}));
  pt_grid gt = g;  // the passes in the plane read K with ky fastest: the table of the cell with x and y exchanged
  std::swap(gt.nx, gt.ny);
  std::swap(gt.L[0], gt.L[1]);
  const float* kt = static_cast<const float*>(kernel_table(ctx, gt, k, PT_FP32));
  // as few tiles as the side allows, all of about the same size (36^3 N = 75: 25 + 25 + 25 instead of 37 + 37 + 1)
  int nb = (N + B - 1) / B, mb = (M + B - 1) / B;
  const std::string name = ctx->tagged("exchange_scratch");
  // A symmetric tile has a field for each of its N^2 slots, though its pairs fill N (N + 1)/2 of them: slots of the triangle
  // alone cost every pass (24^3 N = 16 24.5 -> 25.6 us, 64^3 N = 320 105.5 -> 106.9 ms).  Where the context's HBM budget
  // has no room for them and for those of a batch's other branches, two tiles a side run in the triangle's.
  const size_t branches = size_t(1 + ctx->batch_streams) * (budget / 2);
  const bool tight = sym && nb == 1 && N > 1 && !ctx->fits(name, size_t(N) * N * field, branches);
  if (tight) nb = mb = 2;
  const int bi = (N + nb - 1) / nb, bj = (M + mb - 1) / mb;
  const size_t slots = tight ? size_t(N) * (N + 1) / 2 : size_t(bi) * bj;
  c64* scratch = static_cast<c64*>(ctx->get(name, slots * field));
  for (int J = 0; J * bj < M; ++J)
    for (int I = 0; sym ? I <= J : I * bi < N; ++I) {
      const Tile t{I * bi, std::min(bi, N - I * bi), J * bj, std::min(bj, M - J * bj), int(sym), int(sym && I == J), int(I == 0)};
      if (!fixed_cubic(g)) {
        exchange_tile_axes(g, t, src, tgt, occ, kt, scratch, out, ctx->num_sms, st);
        continue;
      }
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
