// Shifts for the FP64 inverse iteration by bisection, one lane per (k-point, eigenvalue).
//
// The QL iteration runs one k-point per lane: 777 k-points of order 48 are 25 warps, each a serial chain
// of ~3,000 rotations in FP64 (3.6 ms, whatever the rest of the GPU does).  Counting the negative
// pivots of T - x I (Sturm) is the same chain for every x, so here every eigenvalue has a lane of
// its own: W times the parallelism, on the FP32 pipe.  The reported eigenvalues are the FP64 Rayleigh
// quotients of the finished eigenvectors; a shift only has to be close enough to make two
// solves converge: within delta of its eigenvalue, the other vectors' share after two solves is
// (delta / gap)^2.
//   1. FP32 counts: 22 halvings of [-3, 3] (T scaled so that its largest entry is in [1/2, 1)).
//   2. FP32-pair counts (~2^-46 per operation): the bracket is checked, widened if it lost the
//      eigenvalue, and halved to 2^-45.
//   3. Eigenvalues closer than 2^-13 to a neighbour: FP64 counts down to 2^-53, so that delta /
//      gap stays small inside a near-degenerate group too.
#include <algorithm>

#include "fixed.cuh"
#include "kubo_internal.cuh"

namespace kubo {

namespace {

constexpr int BT = 128;
constexpr float PIVMIN32 = 1e-20f;
constexpr double PIVMIN64 = 1e-200;

// negative pivots of T - x I; t4[i] = (d_i, its FP32 remainder, e_(i-1)^2, its remainder)
__device__ __forceinline__ int count32(const float4* t4, int W, float x) {
  int c = 0;
  float q = 1.0f;
  for (int i = 0; i < W; ++i) {
    const float4 a = t4[i];
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
    q = fmaf(-a.z, r, a.x - x);
    if (fabsf(q) < PIVMIN32) q = -PIVMIN32;
    c += q < 0.0f;
  }
  return c;
}

// the same in FP32 pairs: q = (d - x) - e^2 / q, sums by exact TwoSum, the quotient from the
// reciprocal estimate and one exact remainder
__device__ __forceinline__ int count_pair(const float4* t4, int W, float xh, float xl) {
  int c = 0;
  float qh = 1.0f, ql = 0.0f;
  for (int i = 0; i < W; ++i) {
    const float4 a = t4[i];
    float rc;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(qh));
    const float r0 = __fmul_rn(a.z, rc);
    const float rem = fmaf(-r0, ql, __fadd_rn(fmaf(-r0, qh, a.z), a.w));
    const float r1 = __fmul_rn(rem, rc);
    const float s = __fsub_rn(a.x, xh);
    const float b1 = __fsub_rn(s, a.x);
    const float es = __fsub_rn(__fsub_rn(a.x, __fsub_rn(s, b1)), __fadd_rn(xh, b1));
    const float u = __fsub_rn(s, r0);
    const float b2 = __fsub_rn(u, s);
    const float eu = __fsub_rn(__fsub_rn(s, __fsub_rn(u, b2)), __fadd_rn(r0, b2));
    const float l = __fadd_rn(__fadd_rn(__fsub_rn(a.y, xl), es), __fsub_rn(eu, r1));
    qh = __fadd_rn(u, l);
    ql = __fsub_rn(l, __fsub_rn(qh, u));
    if (fabsf(qh) < PIVMIN32) { qh = -PIVMIN32; ql = 0.0f; }
    c += qh < 0.0f;
  }
  return c;
}

__device__ __forceinline__ int count64(const double2* t2, int W, double x) {
  int c = 0;
  double q = 1.0;
  for (int i = 0; i < W; ++i) {
    const double2 a = t2[i];
    q = (a.x - x) - a.y / q;
    if (fabs(q) < PIVMIN64) q = -PIVMIN64;
    c += q < 0.0;
  }
  return c;
}

__global__ void __launch_bounds__(BT) bisect_kernel(int W, int n, int kpc, EighBufs b) {
  extern __shared__ __align__(16) unsigned char bsm[];
  float4* t4 = reinterpret_cast<float4*>(bsm);                                  // [kpc][W]
  double2* t2 = reinterpret_cast<double2*>(t4 + (size_t)kpc * W);               // [kpc][W]
  double* sl = reinterpret_cast<double*>(t2 + (size_t)kpc * W);                 // [kpc][W]
  unsigned* smax = reinterpret_cast<unsigned*>(sl + (size_t)kpc * W);           // [kpc]
  const int t = threadIdx.x;
  const int lk = t / W, j = t - lk * W;
  const int64_t k = (int64_t)blockIdx.x * kpc + lk;
  const bool live = lk < kpc && k < n;
  if (t < kpc) smax[t] = 0u;
  __syncthreads();
  double d = 0.0, e = 0.0;
  if (live) {
    d = b.d[k * W + j];
    e = j > 0 ? b.e[k * W + j - 1] : 0.0;
    atomicMax(&smax[lk], (unsigned)(max(mag_bits(d), mag_bits(e)) >> 32));
  }
  __syncthreads();
  const int ex = live ? (int)(smax[lk] >> 20) - 1022 : 0;   // largest entry below 2^ex
  const bool bad = ex == 0x7FF - 1022;
  if (live) {
    d = bad ? 0.0 : fx::scale_pow2(d, -ex);
    e = bad ? 0.0 : fx::scale_pow2(e, -ex);
    const double e2 = e * e;
    const float dh = (float)d, eh = (float)e2;
    t4[lk * W + j] = make_float4(dh, (float)(d - (double)dh), eh, (float)(e2 - (double)eh));
    t2[lk * W + j] = make_double2(d, e2);
  }
  __syncthreads();
  const float4* T4 = t4 + lk * W;
  const double2* T2 = t2 + lk * W;
  double lam = 0.0;
  if (live) {
    float fl = -3.0f, fh = 3.0f;
#pragma unroll 1
    for (int it = 0; it < 22; ++it) {
      const float m = 0.5f * (fl + fh);
      if (count32(T4, W, m) > j) fh = m;
      else fl = m;
    }
    double lo = (double)fl - 0x1p-19, hi = (double)fh + 0x1p-19;
    auto below = [&](double x) {   // more than j eigenvalues below x
      const float h = (float)x;
      return count_pair(T4, W, h, (float)(x - (double)h)) > j;
    };
    for (double w = 0x1p-17; w < 8.0 && below(lo); w *= 16.0) lo -= w;
    for (double w = 0x1p-17; w < 8.0 && !below(hi); w *= 16.0) hi += w;
#pragma unroll 1
    while (hi - lo > 0x1p-45) {
      const double m = 0.5 * (lo + hi);
      if (below(m)) hi = m;
      else lo = m;
    }
    lam = 0.5 * (lo + hi);
    sl[lk * W + j] = lam;
  }
  __syncthreads();
  if (live) {
    const double* S = sl + lk * W;
    const bool tight = (j > 0 && lam - S[j - 1] < 0x1p-13) || (j + 1 < W && S[j + 1] - lam < 0x1p-13);
    if (tight) {
      double lo = lam - 0x1p-43, hi = lam + 0x1p-43;
      for (double w = 0x1p-42; w < 8.0 && count64(T2, W, lo) > j; w *= 16.0) lo -= w;
      for (double w = 0x1p-42; w < 8.0 && count64(T2, W, hi) <= j; w *= 16.0) hi += w;
#pragma unroll 1
      for (int it = 0; it < 64 && hi - lo > 0x1p-53; ++it) {
        const double m = 0.5 * (lo + hi);
        if (m <= lo || m >= hi) break;   // neighbouring numbers
        if (count64(T2, W, m) > j) hi = m;
        else lo = m;
      }
      lam = 0.5 * (lo + hi);
    }
    // an infinite or NaN entry: NaN for every eigenvalue of the matrix
    b.lam[k * W + j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : fx::scale_pow2(lam, ex);
  }
}

}  // namespace

cudaError_t launch_bisect(int W, int n, EighBufs b, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (W < 1 || W > BT) return cudaErrorInvalidValue;
  const int kpc = BT / W;
  const size_t sm = (size_t)kpc * W * (sizeof(float4) + sizeof(double2) + sizeof(double)) + kpc * sizeof(unsigned);
  bisect_kernel<<<(n + kpc - 1) / kpc, BT, sm, s>>>(W, n, kpc, b);
  return cudaGetLastError();
}

}  // namespace kubo
