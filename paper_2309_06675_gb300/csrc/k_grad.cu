// Reverse mode of steps (1)-(4) (Eq. 2-3): the gradient of L = sum_{e,j} g[e][j] S_e(E_F_j)
// with respect to every entry of H(R), in FP64 grade.
//
// Per k-point, from the forward quantities E, U, v^x = U^dagger dxH U, v^y = U^dagger dyH U:
//   a[e][n]  = sum_j g[e][j] occ_j(E_n) / N_k,   a'[e][n] = sum_j g[e][j] occ_j'(E_n) / N_k
//   num_nm   = -2 Im(v^x_nm v^y_mn),  D^e_nm = (E_n - E_m)^2 + eta_e^2
//   B_nm     = sum_e (a[e][n] - a[e][m]) / D^e_nm                       (antisymmetric)
//   vbar^x   = -i B o v^y,  vbar^y = i B o v^x                          (Hermitian)
//   Ebar_n   = sum_e a'[e][n] Omega^e_n - 2 sum_m (E_n - E_m) num_nm sum_e (a[e][n] - a[e][m]) / (D^e_nm)^2
//   N        = vbar^x v^x + vbar^y v^y
//   Gp       = diag(Ebar) + F o (N^dagger - N),  F_ij = (E_j - E_i) / ((E_j - E_i)^2 + eps^2)
//   Hbar     = U Gp U^dagger,  dxHbar = U vbar^x U^dagger,  dyHbar = U vbar^y U^dagger
// (first-order perturbation theory of the Hermitian eigenproblem for the Gp step), and then
// the transposed Fourier sum
//   G(R) = sum_k e^{-ik.R} [Hbar - i R_x dxHbar - i R_y dyHbar],
// evaluated as one real GEMM over the canonical half set of R: rows (1, cos k.R_h, sin k.R_h)
// against the packed Hermitian columns [Hbar | dxHbar | dyHbar], accumulated over batches in
// a fixed order (deterministic), and unfolded into G(R_h), G(-R_h) = G(R_h)^dagger, G(0).
// This file: the elementwise kernels between the matrix products, which run on the tensor cores in
// FP64 grade (k_zgemm_tc64.cu, k_fourier_tc64.cu).
#include <algorithm>

#include "kubo_internal.cuh"

namespace kubo {

namespace {

constexpr int MAXE = 8;
constexpr int PW = 128;            // threads of the per-k kernels (W <= 128)

// ------------------------------------------------------------------ occupations
__device__ __forceinline__ void occ_and_derivative(double E, double EF, double kT, double& f,
                                                   double& fp) {
  if (kT == 0.0) {
    f = E < EF ? 1.0 : 0.0;
    fp = 0.0;
    return;
  }
  const double x = (E - EF) / kT;
  const double ex = exp(-fabs(x));
  f = x > 0.0 ? ex / (1.0 + ex) : 1.0 / (1.0 + ex);
  fp = -f * (1.0 - f) / kT;
}

// ------------------------------------------------------------------ per-k pair terms
// One CTA per k-point, thread per row p: vbar^x, vbar^y (full W x W) and Ebar.
__global__ void __launch_bounds__(PW) grad_pairs_kernel(
    const double* __restrict__ E, const double2* __restrict__ vx, const double2* __restrict__ vy,
    int W, const double* __restrict__ g, const double* __restrict__ E_F, int n_EF,
    const double* __restrict__ etas, int n_eta, double kT, double inv_Nk,
    double2* __restrict__ vbx, double2* __restrict__ vby, double* __restrict__ Ebar) {
  __shared__ double sE[PW];
  __shared__ double sa[MAXE][PW], sap[MAXE][PW];
  __shared__ double s_emax;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t k = blockIdx.x;
  if (t < W) {
    const double En = E[k * W + t];
    sE[t] = En;
    for (int e = 0; e < n_eta; ++e) {
      double a = 0.0, ap = 0.0;
      for (int j = 0; j < n_EF; ++j) {
        double f, fp;
        occ_and_derivative(En, E_F[j], kT, f, fp);
        const double w = g[e * n_EF + j];
        a = fma(w, f, a);
        ap = fma(w, fp, ap);
      }
      sa[e][t] = a * inv_Nk;
      sap[e][t] = ap * inv_Nk;
    }
  }
  __syncthreads();
  if (warp == 0) {
    double mx = 0.0;
    for (int i = lane; i < W; i += 32) mx = fmax(mx, fabs(sE[i]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) s_emax = mx;
  }
  __syncthreads();
  const int p = t;
  if (p >= W) return;
  const double thr2 = (1e-12 * s_emax) * (1e-12 * s_emax);
  const size_t row = (size_t)k * W * W + (size_t)p * W;
  const double Ep = sE[p];
  double om[MAXE];
#pragma unroll
  for (int e = 0; e < MAXE; ++e) om[e] = 0.0;
  double eb = 0.0;
  for (int m = 0; m < W; ++m) {
    const double2 x = vx[row + m], y = vy[row + m];
    double B = 0.0;
    if (m != p) {
      const double num = -2.0 * (x.y * y.x - x.x * y.y);   // -2 Im(v^x_pm conj(v^y_pm))
      const double dE = Ep - sE[m];
      const double d2 = dE * dE;
      double s2 = 0.0;
#pragma unroll
      for (int e = 0; e < MAXE; ++e) {
        if (e >= n_eta) break;
        const double eta = etas[e];
        if (eta == 0.0 && d2 <= thr2) continue;
        const double D = fma(eta, eta, d2);
        const double iD = 1.0 / D;
        const double da = sa[e][p] - sa[e][m];
        B = fma(da, iD, B);
        s2 = fma(da, iD * iD, s2);
        om[e] = fma(num, iD, om[e]);
      }
      eb = fma(-2.0 * dE * num, s2, eb);
    }
    vbx[row + m] = make_double2(B * y.y, -B * y.x);    // -i B v^y
    vby[row + m] = make_double2(-B * x.y, B * x.x);    //  i B v^x
  }
#pragma unroll
  for (int e = 0; e < MAXE; ++e) {
    if (e >= n_eta) break;
    eb = fma(sap[e][p], om[e], eb);
  }
  Ebar[k * W + p] = eb;
}

// Gp = diag(Ebar) + F o (N^dagger - N), one CTA per k-point
__global__ void __launch_bounds__(256) grad_gp_kernel(const double* __restrict__ E,
                                                      const double* __restrict__ Ebar,
                                                      const double2* __restrict__ N, int W,
                                                      double grad_eps, double2* __restrict__ Gp) {
  __shared__ double sE[PW];
  __shared__ double s_eps2;
  const int t = threadIdx.x;
  const int64_t k = blockIdx.x;
  if (t < W) sE[t] = E[k * W + t];
  __syncthreads();
  if (t == 0) {
    double eps = grad_eps;
    if (!(eps > 0.0)) {
      double mx = 0.0;
      for (int i = 0; i < W; ++i) mx = fmax(mx, fabs(sE[i]));
      eps = 1e-12 * mx;
    }
    s_eps2 = eps * eps;
  }
  __syncthreads();
  const double eps2 = s_eps2;
  const size_t base = (size_t)k * W * W;
  for (int idx = t; idx < W * W; idx += 256) {
    const int i = idx / W, j = idx % W;
    double2 v;
    if (i == j) {
      v = make_double2(Ebar[k * W + i], 0.0);
    } else {
      const double dji = sE[j] - sE[i];
      const double den = fma(dji, dji, eps2);
      const double F = den > 0.0 ? dji / den : 0.0;
      const double2 a = N[base + (size_t)j * W + i], b = N[base + idx];
      v = make_double2(F * (a.x - b.x), F * (-a.y - b.y));   // F (conj(N_ji) - N_ij)
    }
    Gp[base + idx] = v;
  }
}

// Hermitian parts of three full complex matrices -> packed rows [k][3 W^2]
__global__ void pack3_kernel(const double2* __restrict__ A0, const double2* __restrict__ A1,
                             const double2* __restrict__ A2, int W, int n,
                             double* __restrict__ out) {
  const int64_t WW = (int64_t)W * W;
  const int64_t total = (int64_t)n * WW;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = t / WW;
    const int q = (int)(t % WW), i = q / W, j = q % W;
    const int lo = min(i, j), hi = max(i, j);
    const size_t u = (size_t)k * WW + (size_t)lo * W + hi;   // upper element (lo, hi)
    const size_t l = (size_t)k * WW + (size_t)hi * W + lo;   // its mirror
    const double2* src[3] = {A0, A1, A2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double2 x = src[a][u], y = src[a][l];
      // Hermitian part h_lo,hi = (x + conj(y)) / 2: Re above (and on) the diagonal, Im below
      const double v = i <= j ? 0.5 * (x.x + y.x) : 0.5 * (x.y - y.y);
      out[k * 3 * WW + a * WW + q] = v;
    }
  }
}

// unpack element (i, j) of the Hermitian matrix whose packed form is P (W x W reals)
__device__ __forceinline__ double2 herm_at(const double* P, int W, int i, int j) {
  if (i < j) return make_double2(P[i * W + j], P[j * W + i]);
  if (i > j) return make_double2(P[j * W + i], -P[i * W + j]);
  return make_double2(P[i * W + i], 0.0);
}

// G(R) from the accumulated rows: thread per (h or R = 0, i, j)
__global__ void grad_finalize_kernel(const double* __restrict__ Gacc, const int* __restrict__ pairs,
                                     const int* __restrict__ Rh, int idx0, int N_h, int W,
                                     double2* __restrict__ G) {
  const int64_t WW = (int64_t)W * W;
  const int64_t N = 3 * WW;
  const int64_t total = (int64_t)(N_h + 1) * WW;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int h = (int)(t / WW) - 1;
    const int q = (int)(t % WW), i = q / W, j = q % W;
    if (h < 0) {
      G[(size_t)idx0 * WW + q] = herm_at(Gacc, W, i, j);
      continue;
    }
    const double* C = Gacc + (size_t)(1 + h) * N;          // cos row: [CH | CX | CY]
    const double* S = Gacc + (size_t)(1 + N_h + h) * N;    // sin row: [SH | SX | SY]
    const double rx = (double)Rh[3 * h], ry = (double)Rh[3 * h + 1];
    const double2 ch = herm_at(C, W, i, j), cx = herm_at(C + WW, W, i, j), cy = herm_at(C + 2 * WW, W, i, j);
    const double2 sh = herm_at(S, W, i, j), sx = herm_at(S + WW, W, i, j), sy = herm_at(S + 2 * WW, W, i, j);
    // P1 = CH - R_x SX - R_y SY, P2 = SH + R_x CX + R_y CY, G(R_h) = P1 - i P2
    const double2 p1 = make_double2(ch.x - rx * sx.x - ry * sy.x, ch.y - rx * sx.y - ry * sy.y);
    const double2 p2 = make_double2(sh.x + rx * cx.x + ry * cy.x, sh.y + rx * cx.y + ry * cy.y);
    const double2 gv = make_double2(p1.x + p2.y, p1.y - p2.x);
    G[(size_t)pairs[2 * h] * WW + q] = gv;
    G[(size_t)pairs[2 * h + 1] * WW + (size_t)j * W + i] = make_double2(gv.x, -gv.y);   // G(-R) = G(R)^dagger
  }
}

}  // namespace

cudaError_t launch_grad_pairs(const double* E, const double2* vx, const double2* vy, int W, int n,
                              const double* g, const double* E_F, int n_EF, const double* etas,
                              int n_eta, double kT, double inv_Nk, double2* vbx, double2* vby,
                              double* Ebar, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (W > PW || n_eta > MAXE) return cudaErrorInvalidValue;
  grad_pairs_kernel<<<n, PW, 0, s>>>(E, vx, vy, W, g, E_F, n_EF, etas, n_eta, kT, inv_Nk, vbx,
                                     vby, Ebar);
  return cudaGetLastError();
}

cudaError_t launch_grad_gp(const double* E, const double* Ebar, const double2* N, int W, int n,
                           double grad_eps, double2* Gp, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (W > PW) return cudaErrorInvalidValue;
  grad_gp_kernel<<<n, 256, 0, s>>>(E, Ebar, N, W, grad_eps, Gp);
  return cudaGetLastError();
}

cudaError_t launch_pack3(const double2* A0, const double2* A1, const double2* A2, int W, int n,
                         double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t total = (int64_t)n * W * W;
  const int b = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  pack3_kernel<<<b, 256, 0, s>>>(A0, A1, A2, W, n, out);
  return cudaGetLastError();
}

cudaError_t launch_grad_finalize(const double* Gacc, const int* pairs, const int* Rh, int idx0,
                                 int N_h, int W, double2* G, cudaStream_t s) {
  const int64_t total = (int64_t)(N_h + 1) * W * W;
  const int b = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
  grad_finalize_kernel<<<b, 256, 0, s>>>(Gacc, pairs, Rh, idx0, N_h, W, G);
  return cudaGetLastError();
}

}  // namespace kubo
