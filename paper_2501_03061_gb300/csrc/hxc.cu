// Self-consistent local potential of Eq. 1: rho(r) = spin * P(r, r) with P = Phi sigma Phi^*,
// V_Hxc[rho] = V_H + v_xc, V_H the periodic Hartree potential (Poisson equation in G space with the
// G = 0 term removed by the neutralising background) and v_xc the LDA (Slater exchange plus the
// Perdew-Zunger 1981 fit of the Ceperley-Alder correlation energy of the unpolarised gas).
//
// Density: chi = Phi sigma (the library's rotation, tensor cores in the FP32 forms), then
// rho(r) = spin * Re sum_j chi_j(r) conj(phi_j(r)) in one streaming pass over both blocks
// (2 N Ng complex reads, HBM bound), products in the block's precision, sums to 48 bits or more.
// Potential: one FP64 3-D FFT of the real rho, axis by axis on the half spectrum kx <= nx/2: two real rows make
// one complex x line, y and z lines run on nx/2 + 1 columns, the z pass applies 4 pi/|G|^2 / Ng and transforms
// back, and the last x pass evaluates the LDA point by point, adds V_loc and writes the total local potential.
// Small tiles (4 x lines, 8 columns) give every pass 2-4 CTAs per SM: FP64 issues at 1/64 rate, so a pass
// on nz of the 152 SMs is bound by that many FP64 pipes.  60^3: 123 us against 331 us of whole-plane tiles on the
// full spectrum, of which the LDA's transcendentals took 100.  The passes are dependent launches, each reading its
// twiddles while the one before drains: five launches in a row cost small grids more than the three of the whole planes
// (5^3 33 -> 37 us, 60 x 3 x 4 38 -> 48), as dependent ones 29 and 39 (16^3 54 -> 45, 36^3 74 -> 66).
#include <algorithm>

#include "fft.cuh"
#include "internal.h"

namespace pt {

namespace {

constexpr int NT = 64;    // threads per CTA of the FFT passes
constexpr int XL = 4;     // x lines (pairs of rows) per CTA
constexpr int CL = 8;     // columns per CTA of the y and z passes
constexpr int CP = CL + 1;  // their pitch
constexpr double kPi = 3.14159265358979323846;

// Perdew-Zunger correlation of the unpolarised gas (rs >= 1: gamma/(1 + beta1 sqrt(rs) + beta2 rs);
// rs < 1: A ln rs + B + C rs ln rs + D rs) and the Slater exchange; v = d(rho eps)/d rho.
__device__ __forceinline__ void lda_point(double rho, double& eps, double& v) {
  if (!(rho > 1e-30)) {
    eps = 0.0;
    v = 0.0;
    return;
  }
  // t = 1/rs: one cube root serves rs = t^{-1}, sqrt(rs) = t^{-1/2} and (3 rho/pi)^{1/3} = (9/(4 pi^2))^{1/3} t
  constexpr double cx = 0.75 * 0.61088705770857191;  // 3/4 (9/(4 pi^2))^{1/3}
  const double t = cbrt(4.0 * kPi / 3.0 * rho);
  const double ex = -cx * t;
  double ec, vc;
  if (t <= 1.0) {
    const double gamma = -0.1423, b1 = 1.0529, b2 = 0.3334;
    const double s = rsqrt(t), rs = s * s;
    const double inv = 1.0 / (1.0 + b1 * s + b2 * rs);
    ec = gamma * inv;
    vc = ec * (1.0 + (7.0 / 6.0) * b1 * s + (4.0 / 3.0) * b2 * rs) * inv;
  } else {
    const double a = 0.0311, b = -0.048, c = 0.0020, d = -0.0116;
    const double l = -log(t), rs = 1.0 / t;
    ec = a * l + b + c * rs * l + d * rs;
    vc = a * l + (b - a / 3.0) + (2.0 / 3.0) * c * rs * l + (2.0 * d - c) / 3.0 * rs;
  }
  eps = ex + ec;
  v = (4.0 / 3.0) * ex + vc;
}

// running sum of n terms: in FP32 as an unevaluated pair (two-sum: each addition's rounding error is kept, so the
// sum is good to ~n 2^-48), since an FP64 addition of a converted term costs 128 issue cycles on this part
template <class T>
struct RunSum {
  T s = T(0), e = T(0);
  __device__ __forceinline__ void add(T x) {
    if constexpr (sizeof(T) == 8) {
      s += x;
    } else {
      const T n = __fadd_rn(s, x), b = __fsub_rn(n, s);
      e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(n, b)), __fsub_rn(x, b)));
      s = n;
    }
  }
  __device__ __forceinline__ double value() const { return double(s) + double(e); }
};

// the terms of orbitals j, j + 1, ... to the four sums in turn
template <class T, class Sum>
__device__ __forceinline__ double density_sum(const cx<T>* __restrict__ chi, const cx<T>* __restrict__ phi, int N, size_t ng,
                                              size_t r, bool& finite) {
  Sum acc[4];
  int j = 0;
  for (; j + 4 <= N; j += 4) {
    cx<T> a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] = chi[size_t(j + u) * ng + r];
      b[u] = phi[size_t(j + u) * ng + r];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u].add(a[u].re * b[u].re + a[u].im * b[u].im);
  }
  for (; j < N; ++j) {
    const cx<T> a = chi[size_t(j) * ng + r], b = phi[size_t(j) * ng + r];
    acc[0].add(a.re * b.re + a.im * b.im);
  }
  finite = true;
#pragma unroll
  for (int u = 0; u < 4; ++u) finite = finite && isfinite(acc[u].s + acc[u].e);
  return (acc[0].value() + acc[1].value()) + (acc[2].value() + acc[3].value());
}

template <class T>
__global__ void __launch_bounds__(256) k_density(const cx<T>* __restrict__ chi, const cx<T>* __restrict__ phi, int N,
                                                 size_t ng, double spin, double* __restrict__ rho) {
  for (size_t r = size_t(blockIdx.x) * blockDim.x + threadIdx.x; r < ng; r += size_t(gridDim.x) * blockDim.x) {
    bool finite;
    double sum = density_sum<T, RunSum<T>>(chi, phi, N, ng, r, finite);
    // a sum that left the FP32 range, or met a term that is not finite, is taken in FP64
    if (sizeof(T) == 4 && !finite) sum = density_sum<T, RunSum<double>>(chi, phi, N, ng, r, finite);
    rho[r] = spin * sum;
  }
}

// half: [z][y][kx <= nx/2]; rows 2 p and 2 p + 1 of plane z as one complex line
__global__ void __launch_bounds__(NT) k_hxc_x_fwd(GridPlan gp, const double* __restrict__ rho, c128* __restrict__ half,
                                                  const c128* __restrict__ twg) {
  __shared__ c128 tw[kMaxDim];
  __shared__ c128 buf[XL * (kMaxDim + 1)];
  const int z = blockIdx.y, nx = gp.nx, ny = gp.ny, hx = nx / 2 + 1, pitch = gp.pitch_x;
  const int y0 = blockIdx.x * XL * 2;
  for (int t = threadIdx.x; t < nx; t += NT) tw[t] = twg[t];
  pdl_launch_dependents();
  const double* f = rho + (size_t(z) * ny + y0) * nx;
  for (int e = threadIdx.x; e < XL * nx; e += NT) {
    const int l = e / nx, x = e - l * nx, y = y0 + 2 * l;
    buf[l * pitch + x] = c128{y < ny ? f[size_t(2 * l) * nx + x] : 0.0, y + 1 < ny ? f[size_t(2 * l + 1) * nx + x] : 0.0};
  }
  __syncthreads();
  fft_lines<false, NT, XL * kMaxDim>(buf, gp.ax[0], XL, pitch, 1, tw);
  c128* o = half + (size_t(z) * ny + y0) * hx;
  for (int e = threadIdx.x; e < XL * hx; e += NT) {
    const int l = e / hx, k = e - l * hx, y = y0 + 2 * l;
    const c128 u = buf[l * pitch + k], v = buf[l * pitch + (k ? nx - k : 0)];
    // the spectra of the two real rows: Hermitian and anti-Hermitian parts
    if (y < ny) o[size_t(2 * l) * hx + k] = c128{0.5 * (u.re + v.re), 0.5 * (u.im - v.im)};
    if (y + 1 < ny) o[size_t(2 * l + 1) * hx + k] = c128{0.5 * (u.im + v.im), 0.5 * (v.re - u.re)};
  }
}

// y lines of the half spectrum in place
template <bool INV>
__global__ void __launch_bounds__(NT) k_hxc_y(GridPlan gp, c128* __restrict__ half, const c128* __restrict__ twg) {
  __shared__ c128 tw[kMaxDim];
  __shared__ c128 buf[CP * kMaxDim];
  const int ny = gp.ny, hx = gp.nx / 2 + 1, k0 = blockIdx.x * CL, cols = min(CL, hx - k0);
  for (int t = threadIdx.x; t < ny; t += NT) tw[t] = twg[gp.nx + t];
  pdl_wait();  // the pass before
  pdl_launch_dependents();
  c128* f = half + size_t(blockIdx.y) * ny * hx + k0;
  for (int e = threadIdx.x; e < CL * ny; e += NT) {
    const int y = e / CL, c = e % CL;
    if (c < cols) buf[y * CP + c] = f[size_t(y) * hx + c];
  }
  __syncthreads();
  fft_lines<INV, NT, CL * kMaxDim>(buf, gp.ax[1], cols, 1, CP, tw);
  for (int e = threadIdx.x; e < CL * ny; e += NT) {
    const int y = e / CL, c = e % CL;
    if (c < cols) f[size_t(y) * hx + c] = buf[y * CP + c];
  }
}

// z lines: forward, times 4 pi/|G|^2 / Ng, inverse, in place
__global__ void __launch_bounds__(NT) k_hxc_z(GridPlan gp, c128* __restrict__ half, const double* __restrict__ g2,
                                              double inv_ng, const c128* __restrict__ twg) {
  __shared__ c128 tw[kMaxDim];
  __shared__ c128 buf[CP * kMaxDim];
  const int nx = gp.nx, ny = gp.ny, nz = gp.nz, hx = nx / 2 + 1, y = blockIdx.y;
  const int k0 = blockIdx.x * CL, cols = min(CL, hx - k0);
  for (int t = threadIdx.x; t < nz; t += NT) tw[t] = twg[nx + ny + t];
  pdl_wait();  // the pass before
  pdl_launch_dependents();
  c128* f = half + size_t(y) * hx + k0;
  for (int e = threadIdx.x; e < CL * nz; e += NT) {
    const int z = e / CL, c = e % CL;
    if (c < cols) buf[z * CP + c] = f[size_t(z) * ny * hx + c];
  }
  __syncthreads();
  fft_lines<false, NT, CL * kMaxDim>(buf, gp.ax[2], cols, 1, CP, tw);
  for (int e = threadIdx.x; e < CL * nz; e += NT) {
    const int z = e / CL, c = e % CL;
    if (c >= cols) continue;
    const double G2 = g2[k0 + c] + g2[nx + y] + g2[nx + ny + z];
    buf[z * CP + c] = buf[z * CP + c] * (G2 > 0.0 ? 4.0 * kPi / G2 * inv_ng : 0.0);
  }
  __syncthreads();
  fft_lines<true, NT, CL * kMaxDim>(buf, gp.ax[2], cols, 1, CP, tw);
  for (int e = threadIdx.x; e < CL * nz; e += NT) {
    const int z = e / CL, c = e % CL;
    if (c < cols) f[size_t(z) * ny * hx + c] = buf[z * CP + c];
  }
}

// inverse x lines (two rows per complex line), LDA, V_loc; optional energy sums of the CTA's rows, part[2 cta + {0, 1}]
__global__ void __launch_bounds__(NT) k_hxc_x_inv(GridPlan gp, const c128* __restrict__ half, const double* __restrict__ rho,
                                                  const double* __restrict__ vloc, double* __restrict__ vout,
                                                  double* __restrict__ part, const c128* __restrict__ twg) {
  __shared__ c128 tw[kMaxDim];
  __shared__ c128 buf[XL * (kMaxDim + 1)];
  __shared__ double red[2][NT / 32];
  const int z = blockIdx.y, nx = gp.nx, ny = gp.ny, hx = nx / 2 + 1, pitch = gp.pitch_x;
  const int y0 = blockIdx.x * XL * 2;
  for (int t = threadIdx.x; t < nx; t += NT) tw[t] = twg[t];
  pdl_wait();  // the pass before
  pdl_launch_dependents();
  const c128* f = half + (size_t(z) * ny + y0) * hx;
  for (int e = threadIdx.x; e < XL * hx; e += NT) {
    const int l = e / hx, k = e - l * hx, y = y0 + 2 * l;
    const c128 a = y < ny ? f[size_t(2 * l) * hx + k] : czero<double>();
    const c128 b = y + 1 < ny ? f[size_t(2 * l + 1) * hx + k] : czero<double>();
    buf[l * pitch + k] = c128{a.re - b.im, a.im + b.re};                     // a + i b
    if (k && 2 * k != nx) buf[l * pitch + nx - k] = c128{a.re + b.im, b.re - a.im};  // conj(a) + i conj(b)
  }
  __syncthreads();
  fft_lines<true, NT, XL * kMaxDim>(buf, gp.ax[0], XL, pitch, 1, tw);
  const size_t off = (size_t(z) * ny + y0) * nx;
  const int rows = min(2 * XL, ny - y0);
  double eh = 0.0, exc = 0.0;
  for (int e = threadIdx.x; e < rows * nx; e += NT) {
    const int q = e / nx, x = e - q * nx;
    const c128 w = buf[(q >> 1) * pitch + x];
    const double vh = q & 1 ? w.im : w.re;
    const double r = rho[off + e];
    double eps, vxc;
    lda_point(r, eps, vxc);
    vout[off + e] = (vloc ? vloc[off + e] : 0.0) + vh + vxc;
    eh += 0.5 * r * vh;
    exc += r * eps;
  }
  if (!part) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    eh += __shfl_xor_sync(0xffffffffu, eh, o);
    exc += __shfl_xor_sync(0xffffffffu, exc, o);
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = eh;
    red[1][w] = exc;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    double a = 0.0;
    for (int k = 0; k < NT / 32; ++k) a += red[threadIdx.x][k];
    part[2 * (size_t(z) * gridDim.x + blockIdx.x) + threadIdx.x] = a;
  }
}

// out[2 z + {0, 1}]: the sums of plane z's CTAs
__global__ void k_hxc_energy(const double* __restrict__ part, int per_plane, int nz, double* __restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2 * nz) return;
  double a = 0.0;
  for (int k = 0; k < per_plane; ++k) a += part[2 * (size_t(e >> 1) * per_plane + k) + (e & 1)];
  out[e] = a;
}

}  // namespace

template <class T>
void density(pt_ctx* ctx, const cx<T>* phi, const c128* sigma, int N, size_t ng, double spin, cx<T>* chi,
             double* rho, cudaStream_t st) {
  // chi_j = sum_i sigma_ij phi_i
  rotate<T>(ctx, phi, sigma, N, N, N, ng, c128{1.0, 0.0}, nullptr, 0, chi, st);
  const int blocks = int(std::max<size_t>(1, std::min<size_t>((ng + 255) / 256, size_t(ctx->num_sms) * 16)));
  PT_LAUNCH(k_density<T>, blocks, 256, 0, st, chi, phi, N, ng, spin, rho);
}

template void density<float>(pt_ctx*, const c64*, const c128*, int, size_t, double, c64*, double*, cudaStream_t);
template void density<double>(pt_ctx*, const c128*, const c128*, int, size_t, double, c128*, double*, cudaStream_t);

void hxc_potential(pt_ctx* ctx, const double* rho, const double* vloc, const pt_grid& g, double* v, double* part,
                   cudaStream_t st) {
  const FftTables& ft = fft_tables(ctx, g, PT_FP64);
  const size_t ng = ng_of(g);
  const int hx = g.nx / 2 + 1, xc = (g.ny + 2 * XL - 1) / (2 * XL), cc = (hx + CL - 1) / CL;
  // the half spectrum, and per-CTA energy sums
  const size_t nh = size_t(hx) * g.ny * g.nz;
  c128* half = static_cast<c128*>(ctx->get("hxc_scratch", nh * sizeof(c128) + 2 * size_t(xc) * g.nz * sizeof(double)));
  double* sums = part ? reinterpret_cast<double*>(half + nh) : nullptr;
  const c128* tw = static_cast<const c128*>(ft.tw);
  // Launched dependent, the CTAs of a pass settle where the pass before leaves room.  With more than two a SM in both of two
  // passes that leaves some SMs with twice the work of others (64^3 130 -> 158 us; 64 x 60 x 60, 300 CTAs a pass, 129
  // -> 121): those run one after another.
  const int two = 2 * ctx->num_sms;
  const bool crowded = cc * g.ny > two && cc * g.nz > two;
  auto next = [&](auto kernel, dim3 grid, auto... args) {
    if (crowded) PT_LAUNCH(kernel, grid, NT, 0, st, args...);
    else PT_LAUNCH_PDL(kernel, grid, NT, 0, st, args...);
  };
  const double* g2 = static_cast<const double*>(ft.g2d);
  PT_LAUNCH(k_hxc_x_fwd, dim3(xc, g.nz), NT, 0, st, ft.plan, rho, half, tw);
  next(k_hxc_y<false>, dim3(cc, g.nz), ft.plan, half, tw);
  next(k_hxc_z, dim3(cc, g.ny), ft.plan, half, g2, 1.0 / double(ng), tw);
  next(k_hxc_y<true>, dim3(cc, g.nz), ft.plan, half, tw);
  next(k_hxc_x_inv, dim3(xc, g.nz), ft.plan, half, rho, vloc, v, sums, tw);
  if (part) PT_LAUNCH(k_hxc_energy, (2 * g.nz + 127) / 128, 128, 0, st, sums, xc, g.nz, part);
}

}  // namespace pt
