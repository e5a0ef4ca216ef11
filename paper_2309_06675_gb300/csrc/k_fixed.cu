// FP64-grade matrix work of steps (2)-(4) on the integer pipe (fixed.cuh):
//
//   berry_fix_kernel   v^a = U^dagger (d_a H) U for a = x, y and the curvature of Eq. 3 (W <= 24; to 64
//                      where a caller's workspace has no room for k_zgemm_tc64.cu's matrices)
//   reflect_fix_kernel U = Q D Z: the Householder reflectors applied to the eigenvectors of T
//
// Both were FP64 kernels at 85-96 % of the FP64 pipe; the products here are sums of 59-bit
// fixed-point products, five times as many per clock.  Energy differences, curvature quotients
// and the band sums stay FP64.
#include <algorithm>

#include "fixed.cuh"
#include "kubo_internal.cuh"

namespace kubo {

namespace {

#ifndef BERRY_FEW
#define BERRY_FEW 608
#endif
constexpr int MAXE = 8;
constexpr int EXP_BAD = 1 << 20;   // operand with an infinite or NaN entry: the results are NaN

// A k-point's value into its shared-memory word (by every thread of the CTA).  Where the CTA is one k-point each
// warp adds up first: a 64-bit atomic on one word takes its lanes one after the other (one matrix of W = 16 by 256 threads:
// the kernel 40 us, 17 with this).
template <class Op, class Put>
__device__ __forceinline__ void add_up(bool whole, unsigned long long v, Op op, Put put) {
  if (whole) {
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v) put(v);
  } else if (v) {
    put(v);
  }
}

// ------------------------------------------------------------------ rotations and curvature
// KPC k-points per CTA, nthr = NX x NY threads each; thread (ty, tx) owns the outputs (ty + NY i,
// tx + NX j) of the W x W products, i < TM, j < TN (rows and columns beyond W repeat the last one and
// are dropped).  Per k-point in shared memory: U and dH (then T = dH U in its place) as limbs
// [W][LD], v^x of the thread's own pairs, energies.  Products whose pair n < m lies entirely below the
// diagonal are skipped at compile time when NX = 2 NY (TM = 4, TN = 2) or NX = NY (TM = TN).
//
// Scales: dH by 2^-e with 2^e above its Frobenius norm, so rows, T = dH U and v = U^dagger T stay
// below 1 by Cauchy-Schwarz; U by 2^-ue (58 fractional bits; ue = null: unit columns).
template <int TM, int TN>
__global__ void __launch_bounds__(512, 1)
    berry_fix_kernel(const double* __restrict__ E, const double2* __restrict__ U,
                     const double* __restrict__ Xp, const double* __restrict__ Yp, int64_t ld,
                     int W, int n, const double* __restrict__ etas, int n_eta,
                     double* __restrict__ Om, int64_t eta_stride, int NX, int NY, int KPC, int LD,
                     const int* __restrict__ ue) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NO = TM * TN;
  const int t = threadIdx.x;
  const int nthr = NX * NY;
  const int lk = t / nthr, r0 = t - lk * nthr;
  const int ty = r0 / NX, tx = r0 - ty * NX;
  const int64_t k = (int64_t)blockIdx.x * KPC + lk;
  const bool live = lk < KPC && k < n;
  int4* sUall = reinterpret_cast<int4*>(smraw);
  int4* sAall = sUall + (size_t)KPC * W * LD;
  double2* sV = reinterpret_cast<double2*>(sAall + (size_t)KPC * W * LD);   // [NO][blockDim]
  double* sEall = reinterpret_cast<double*>(sV + (size_t)NO * blockDim.x);
  unsigned long long* sq = reinterpret_cast<unsigned long long*>(sEall + (size_t)KPC * W);   // [KPC]
  unsigned long long* semax = sq + KPC;                                                     // [KPC]
  unsigned* smax = reinterpret_cast<unsigned*>(semax + KPC);                                // [KPC]
  const int lkc = lk < KPC ? lk : 0;
  int4* sU = sUall + (size_t)lkc * W * LD;
  int4* sA = sAall + (size_t)lkc * W * LD;
  double* sE = sEall + lkc * W;
  const int WW = W * W;
  const FastDiv dW(W);

  for (int i = t; i < KPC; i += blockDim.x) semax[i] = 0ull;
  __syncthreads();
  int eu = 0;
  unsigned long long top = 0ull;
  if (live) {
    eu = ue ? ue[k] : 0;
    const double2* Uk = U + (size_t)k * WW;
    for (int idx = r0; idx < WW; idx += nthr) {
      const int r = (int)dW.div(idx), c = idx - r * W;
      const double2 u = Uk[idx];
      sU[r * LD + c] = eu == EXP_BAD ? make_int4(0, 0, 0, 0)
                                     : fx::climbs(fx::from_double(u.x, 58 - eu), fx::from_double(u.y, 58 - eu));
    }
    for (int j = r0; j < W; j += nthr) {
      const double e = E[k * W + j];
      sE[j] = e;
      const unsigned long long m = mag_bits(e);
      if (m <= 0x7FF0000000000000ull) top = max(top, m);
    }
  }
  add_up(KPC == 1, top, [](unsigned long long a, unsigned long long b) { return max(a, b); },
         [&](unsigned long long v) { atomicMax(&semax[lkc], v); });
  int row[TM], col[TN];
#pragma unroll
  for (int i = 0; i < TM; ++i) row[i] = min(ty + NY * i, W - 1);
#pragma unroll
  for (int j = 0; j < TN; ++j) col[j] = min(tx + NX * j, W - 1);

  int ex[2];
  double num[TM][TN];
#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir) {
    // ---- dH: exponent of its Frobenius norm, then limbs of the full Hermitian matrix
    if (t < KPC) { sq[t] = 0ull; smax[t] = 0u; }
    __syncthreads();   // (also: the previous direction's reads of sA are done)
    const double* P = (dir == 0 ? Xp : Yp) + (live ? k : 0) * ld;
    double v[NO];
    unsigned mx = 0u;
#pragma unroll
    for (int q = 0; q < NO; ++q) {   // NO x nthr >= W^2
      const int idx = r0 + q * nthr;
      v[q] = live && idx < WW ? P[idx] : 0.0;
      mx = max(mx, (unsigned)(mag_bits(v[q]) >> 32));
    }
    if (live && mx) atomicMax(&smax[lkc], mx);
    __syncthreads();
    const int emax = (int)(smax[lkc] >> 20);   // biased exponent of the largest entry
    {
      unsigned long long s = 0ull;
#pragma unroll
      for (int q = 0; q < NO; ++q) {
        const int idx = r0 + q * nthr;
        const int i = (int)dW.div(idx), j = idx - i * W;
        const unsigned hi = (unsigned)(mag_bits(v[q]) >> 32);
        const int sh = emax - (int)(hi >> 20);
        // |v| below (m + 1) 2^(emax - 14), m the leading 15 bits at the common exponent
        const unsigned m = hi && sh < 15 ? ((((hi & 0xFFFFFu) | 0x100000u) >> 6) >> sh) : 0u;
        if (idx < WW && hi) s += (unsigned long long)((m + 1) * (m + 1)) << (i == j ? 0 : 1);
      }
      add_up(KPC == 1, s, [](unsigned long long a, unsigned long long b) { return a + b; },
             [&](unsigned long long v) { atomicAdd(&sq[lkc], v); });   // (0 where not live)
    }
    __syncthreads();
    // 2^e above the norm: norm^2 <= sq 2^(2 (emax - 1023 - 14)), sq < 2^(63 - clz + 1)
    const unsigned long long s2 = sq[lkc];
    const int e = emax == 0x7FF || eu == EXP_BAD ? EXP_BAD
                  : s2 == 0ull ? 0 : emax - 1023 - 14 + ((64 - __clzll((long long)s2) + 1) >> 1);
    ex[dir] = e;
    if (live) {
#pragma unroll
      for (int q = 0; q < NO; ++q) {
        const int idx = r0 + q * nthr;
        if (idx >= WW) break;
        const int i = (int)dW.div(idx), j = idx - i * W;
        const int2 l = e == EXP_BAD ? make_int2(0, 0) : fx::limbs(fx::from_double(v[q], fx::BITS - e));
        // packed entry (i <= j): Re of (i, j) and (j, i); (i > j): Im of (j, i), minus that of (i, j)
        int2* a = reinterpret_cast<int2*>(sA + i * LD + j);
        int2* b = reinterpret_cast<int2*>(sA + j * LD + i);
        if (i < j) { a[0] = l; b[0] = l; }
        else if (i > j) { b[1] = l; a[1] = make_int2(-l.x, -l.y); }
        else { a[0] = l; a[1] = make_int2(0, 0); }
      }
    }
    __syncthreads();
    // ---- T = dH U (58 + 59 fractional bits folded back to 59)
    fx::Acc acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) fx::zero(acc[i][j]);
    if (live)
#pragma unroll 1
      for (int q = 0; q < W; ++q) {
        int4 b[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) b[j] = sU[q * LD + col[j]];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const int4 a = sA[row[i] * LD + q];
          const int nh = -a.z, nl = -a.w;
#pragma unroll
          for (int j = 0; j < TN; ++j) fx::cmad(acc[i][j], a, nh, nl, b[j]);
        }
      }
    __syncthreads();
    if (live)
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j)
          if (ty + NY * i < W && tx + NX * j < W)
            sA[row[i] * LD + col[j]] = fx::climbs(fx::fold_shift(acc[i][j].rh, acc[i][j].rm, 2),
                                                  fx::fold_shift(acc[i][j].ih, acc[i][j].im, 2));
    __syncthreads();
    // ---- v = U^dagger T, the pairs n < m only
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) fx::zero(acc[i][j]);
    if (live)
#pragma unroll 1
      for (int q = 0; q < W; ++q) {
        int4 b[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) b[j] = sA[q * LD + col[j]];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const int4 a = sU[q * LD + row[i]];
          const int nh = -a.z, nl = -a.w;
#pragma unroll
          for (int j = 0; j < TN; ++j)
            // rows >= NY i, columns < NX (j + 1): all pairs below the diagonal
            if (TN * i < TM * (j + 1)) fx::cmadc(acc[i][j], a, nh, nl, b[j]);
        }
      }
    // v = fold 2^(e + 2 ue - 61); the power of two enters with the pair's numerator
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        if (!(TN * i < TM * (j + 1))) continue;
        const double2 w = make_double2((double)fx::fold(acc[i][j].rh, acc[i][j].rm),
                                       (double)fx::fold(acc[i][j].ih, acc[i][j].im));
        if (dir == 0) {
          sV[(i * TN + j) * blockDim.x + t] = w;   // read back by this thread only
        } else {
          const double2 x = sV[(i * TN + j) * blockDim.x + t];
          num[i][j] = -2.0 * (x.y * w.x - x.x * w.y);
        }
      }
  }
  // ---- Omega_n = sum_m T_nm, every pair once: +T to n, -T to m (exactly antisymmetric)
  const bool bad = ex[0] == EXP_BAD || ex[1] == EXP_BAD;
  const int es = bad ? 0 : ex[0] + ex[1] + 4 * eu - 122;
  const double emaxE = __longlong_as_double((long long)semax[lkc]);
  const double thr2 = (1e-12 * emaxE) * (1e-12 * emaxE);
  unsigned pairs = 0u;
  double d2[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      d2[i][j] = 0.0;
      const int a = ty + NY * i, b = tx + NX * j;
      if (!(TN * i < TM * (j + 1)) || !live || a >= b || b >= W) continue;
      pairs |= 1u << (i * TN + j);
      num[i][j] = bad ? __longlong_as_double(0x7FF8000000000000ll) : fx::scale_pow2(num[i][j], es);
      const double dE = sE[a] - sE[b];
      d2[i][j] = dE * dE;
    }
  // partial sums [W][NX + NY] per k-point in the place of T
  double* red = reinterpret_cast<double*>(sA);
  const int LR = NX + NY;
#pragma unroll 1
  for (int e = 0; e < n_eta; ++e) {
    const double eta = etas[e];
    const bool eta0 = eta == 0.0;
    double rp[TM], cp[TN];
#pragma unroll
    for (int i = 0; i < TM; ++i) rp[i] = 0.0;
#pragma unroll
    for (int j = 0; j < TN; ++j) cp[j] = 0.0;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        if (!(TN * i < TM * (j + 1)) || !((pairs >> (i * TN + j)) & 1u)) continue;
        if (eta0 && d2[i][j] <= thr2) continue;
        const double T = num[i][j] / fma(eta, eta, d2[i][j]);
        rp[i] += T;
        cp[j] -= T;
      }
    __syncthreads();   // the reads of sA (e = 0) or of the previous partial sums are done
    if (live) {
#pragma unroll
      for (int i = 0; i < TM; ++i)
        if (ty + NY * i < W) red[(ty + NY * i) * LR + tx] = rp[i];
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (tx + NX * j < W) red[(tx + NX * j) * LR + NX + ty] = cp[j];
    }
    __syncthreads();
    if (live)
      for (int a = r0; a < W; a += nthr) {
        double s = 0.0;
        for (int q = 0; q < LR; ++q) s += red[a * LR + q];
        Om[e * eta_stride + k * W + a] = s;
      }
  }
}

// per-matrix exponent with every column norm of U below 2^ue (1 + 2^-34), for eigenvectors supplied by the
// caller; warp per column in turn, CTA per matrix.  (The tolerance keeps ue = 0, and with it the last bit, for
// unit columns with the rounding of any eigensolver.  It is below what dH's scale leaves over: the leading 15
// bits of one dominating diagonal entry and a unit for each other one keep a row's norm below 1 - 2^-31, and rows
// of several large entries stay further below their matrix's Frobenius norm, so |T| < 1.)
__global__ void __launch_bounds__(256) unorm_kernel(const double2* __restrict__ U, int W,
                                                    int* __restrict__ ue) {
  __shared__ int s_e;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const double2* Uk = U + (size_t)blockIdx.x * W * W;
  if (t == 0) s_e = -4096;
  __syncthreads();
  int em = -4096;
  for (int c = warp; c < W; c += 8) {
    unsigned mx = 0u;
    for (int r = lane; r < W; r += 32) {
      const double2 u = Uk[(size_t)r * W + c];
      mx = max(mx, (unsigned)(max(mag_bits(u.x), mag_bits(u.y)) >> 32));
    }
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int ex = (int)(mx >> 20);
    if (ex == 0x7FF) { em = EXP_BAD; break; }
    if (ex == 0) continue;   // zeros and subnormals
    // squares at the column's own exponent
    double s = 0.0;
    for (int r = lane; r < W; r += 32) {
      const double2 u = Uk[(size_t)r * W + c];
      const double a = fx::scale_pow2(u.x, 1023 - ex), b = fx::scale_pow2(u.y, 1023 - ex);
      s = fma(a, a, fma(b, b, s));
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    // norm = sqrt(s) 2^(ex - 1023)
    int f = 0;
    frexp(sqrt(s) * (1.0 - 0x1p-34), &f);   // < 2^f
    em = max(em, f + ex - 1023);
  }
  if (lane == 0) atomicMax(&s_e, em);
  __syncthreads();
  if (t == 0) ue[blockIdx.x] = s_e >= 900 ? EXP_BAD : s_e < -900 ? 0 : s_e;
}

// ------------------------------------------------------------------ U = Q D Z
// One k-point (above W = 64: half of its columns) per CTA: u (limbs, 58 fractional bits) starts as
// its columns of D Z; the unit reflectors
// w_j = v_j sqrt(tau_j / 2), H_j = I - 2 w_j w_j^dagger, are applied four at a time from the last:
//   s_a = w_a^dagger u,   h_a = s_a - 2 sum_{b > a} (w_a^dagger w_b) h_b,   u -= 2 sum_a w_a h_a,
// which is H_j0 H_j0+1 H_j0+2 H_j0+3 u with one pass for the four sums and one for the update (a
// triangular factor as in the compact WY form would need more range than the h_a, each at most
// 1).  Four lanes share the rows of a column.
// What bounds it: the 24 integer multiply-adds per element and reflector, each four cycles of a
// sub-core's multiplier (80 % busy at W = 64): 4,096 k-points take 2.55 ms, with the update's operands pinned
// (fixed.cuh); 3.4 before that.
constexpr int RF_NT = 256;
constexpr int RF_NB = 4;

__host__ __device__ __forceinline__ int rf_blocks(int W) { return W > 2 ? (W - 2 + RF_NB - 1) / RF_NB : 0; }

__global__ void __launch_bounds__(RF_NT, 2)
    reflect_fix_kernel(int W, EighBufs b, const double* __restrict__ Z, double2* __restrict__ Uout,
                       int CB, int LD) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int4* su = reinterpret_cast<int4*>(smraw);              // [W][LD], CB columns
  int4* sw = su + (size_t)W * LD;                         // 2 x [W][RF_NB]: a block's reflectors by rows
  int4* sg = sw + (size_t)2 * W * RF_NB;                  // 2 x [6] w_a^dagger w_b
  int4* sp = sg + 12;                                     // [W] phases
  double* sf = reinterpret_cast<double*>(sp + W);         // [W] sqrt(tau / 2)
  const int t = threadIdx.x, q = t & 3, nt = blockDim.x;
  const int64_t k = blockIdx.x;
  const double* Zk = Z + (size_t)k * W * W;
  const double2* R = b.refl + (size_t)k * W * W;
  const int cb0 = blockIdx.y * CB, ncol = min(CB, W - cb0);
  const FastDiv dC(ncol);
  for (int j = t; j < W; j += nt) {
    const double2 p = b.phase[k * W + j];
    sp[j] = fx::climbs(fx::from_double(p.x, 58), fx::from_double(p.y, 58));
    sf[j] = sqrt(0.5 * b.tau[k * W + j]);
  }
  // (a column of Z with a NaN is NaN throughout, from its normalisation: the first row tells)
  const bool any_bad = __syncthreads_or(t < ncol && !fx::finite(Zk[cb0 + t]));
  for (int idx = t; idx < W * ncol; idx += nt) {
    const int r = (int)dC.div(idx), c = idx - r * ncol;
    const int2 z = fx::limbs(fx::from_double(Zk[(size_t)r * W + cb0 + c], 58));
    const int4 p = sp[r];
    long long rh = 0, rm = 0, ih = 0, im = 0;
    fx::mad(rh, p.x, z.x); fx::mad(rm, p.x, z.y); fx::mad(rm, p.y, z.x);
    fx::mad(ih, p.z, z.x); fx::mad(im, p.z, z.y); fx::mad(im, p.w, z.x);
    su[r * LD + c] = fx::climbs(fx::fold_shift(rh, rm, 2), fx::fold_shift(ih, im, 2));
  }
  const int nblk = rf_blocks(W), nref = W - 2;
  // stage block bk: rows j0 + 1 .. W - 1 of its reflectors (zero above each one's first row)
  auto stage = [&](int bk, int buf) {
    const int j0 = bk * RF_NB;
    for (int idx = t; idx < (W - j0 - 1) * RF_NB; idx += nt) {
      const int r = j0 + 1 + (idx >> 2), a = idx & 3, j = j0 + a;
      int4 w = make_int4(0, 0, 0, 0);
      if (j < nref && r > j) {
        const double f = sf[j];
        const double2 v = R[(size_t)r * W + j];
        w = fx::climbs(fx::from_double(v.x * f, 58), fx::from_double(v.y * f, 58));
      }
      sw[(size_t)buf * W * RF_NB + r * RF_NB + a] = w;
    }
  };
  // g_ab = w_a^dagger w_b of the staged block, a warp per pair (58 fractional bits)
  auto gram = [&](int bk, int buf) {
    const int lane = t & 31;
    const int4* w = sw + (size_t)buf * W * RF_NB;
    for (int p = t >> 5; p < 6; p += nt >> 5) {
      const int a = p < 3 ? 0 : p < 5 ? 1 : 2;
      const int c = p < 3 ? p + 1 : p < 5 ? p - 1 : 3;
      fx::Acc acc;
      fx::zero(acc);
      for (int r = bk * RF_NB + 1 + lane; r < W; r += 32) {
        const int4 x = w[r * RF_NB + a], y = w[r * RF_NB + c];
        fx::cmadc(acc, x, -x.z, -x.w, y);
      }
      long long re = fx::fold(acc.rh, acc.rm), im = fx::fold(acc.ih, acc.im);   // units 2^-60
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) sg[buf * 6 + p] = fx::climbs(fx::rshift(re, 2), fx::rshift(im, 2));
    }
  };
  if (nblk > 0) {
    stage(nblk - 1, (nblk - 1) & 1);
    __syncthreads();
    gram(nblk - 1, (nblk - 1) & 1);
  }
  __syncthreads();
#pragma unroll 1
  for (int bk = nblk - 1; bk >= 0; --bk) {
    const int buf = bk & 1, j0 = bk * RF_NB;
    if (bk > 0) stage(bk - 1, buf ^ 1);
    const int4* w = sw + (size_t)buf * W * RF_NB;
    for (int c0 = 0; c0 < ncol; c0 += nt >> 2) {
      const int c = min(c0 + (t >> 2), ncol - 1);
      const bool act = c0 + (t >> 2) < ncol;
      fx::Acc s[RF_NB];
#pragma unroll
      for (int a = 0; a < RF_NB; ++a) fx::zero(s[a]);
#pragma unroll 1
      for (int r = j0 + 1 + q; r < W; r += 4) {
        const int4 u = su[r * LD + c];
        const int nh = -u.z, nl = -u.w;
#pragma unroll
        for (int a = 0; a < RF_NB; ++a) {
          // conj(w) u; its imaginary part w_x u_y - w_y u_x negated, so that one negation (of
          // Im u) serves the four products
          const int4 x = w[r * RF_NB + a];
          fx::mad(s[a].rh, x.x, u.x); fx::mad(s[a].rm, x.x, u.y); fx::mad(s[a].rm, x.y, u.x);
          fx::mad(s[a].rh, x.z, u.z); fx::mad(s[a].rm, x.z, u.w); fx::mad(s[a].rm, x.w, u.z);
          fx::mad(s[a].ih, x.x, nh); fx::mad(s[a].im, x.x, nl); fx::mad(s[a].im, x.y, nh);
          fx::mad(s[a].ih, x.z, u.x); fx::mad(s[a].im, x.z, u.y); fx::mad(s[a].im, x.w, u.x);
        }
      }
      int4 h[RF_NB];   // -h_a
#pragma unroll
      for (int a = RF_NB - 1; a >= 0; --a) {
        long long re = -fx::fold(s[a].rh, s[a].rm), im = fx::fold(s[a].ih, s[a].im);   // -s, units 2^-60
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          re += __shfl_xor_sync(0xffffffffu, re, o);
          im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        fx::Acc c2;
        fx::zero(c2);
#pragma unroll
        for (int b2 = a + 1; b2 < RF_NB; ++b2) {
          const int4 g = sg[buf * 6 + (a == 0 ? b2 - 1 : a == 1 ? b2 + 1 : 5)];
          fx::cmad(c2, g, -g.z, -g.w, h[b2]);
        }
        h[a] = fx::climbs(fx::rshift(re - 2 * fx::fold(c2.rh, c2.rm), 2),
                          fx::rshift(im - 2 * fx::fold(c2.ih, c2.im), 2));
      }
      if (act)
#pragma unroll 1
        for (int r = j0 + 1 + q; r < W; r += 4) {
          // u + sum w (-h) / 2, rounded once: the sums start at 2 u and the half
          const int4 u = su[r * LD + c];
          fx::Acc d;
          d.rh = (long long)u.x * (1 << (fx::LB + 1)) + (2 * u.y + 1);
          d.ih = (long long)u.z * (1 << (fx::LB + 1)) + (2 * u.w + 1);
          d.rm = d.im = 0;
#pragma unroll
          for (int a = 0; a < RF_NB; ++a) {
            const int4 x = w[r * RF_NB + a];
            fx::cmad(d, x, -x.z, -x.w, fx::pin(h[a]));
          }
          su[r * LD + c] = fx::climbs((d.rh + (d.rm >> fx::LB)) >> 1, (d.ih + (d.im >> fx::LB)) >> 1);
        }
    }
    __syncthreads();
    if (bk > 0) gram(bk - 1, buf ^ 1);
    __syncthreads();
  }
  double2* Uk = Uout + (size_t)k * W * W;
  for (int idx = t; idx < W * ncol; idx += nt) {
    const int r = (int)dC.div(idx), c = idx - r * ncol;
    const int4 u = su[r * LD + c];
    double2 v = make_double2(fx::to_double(fx::value(u.x, u.y), -58), fx::to_double(fx::value(u.z, u.w), -58));
    if (any_bad && !fx::finite(Zk[cb0 + c])) v.x = v.y = __longlong_as_double(0x7FF8000000000000ll);
    Uk[(size_t)r * W + cb0 + c] = v;
  }
}

// U = Q D Z for W <= 16: a thread per column of a k-point, its column in registers (limbs), 256 / W
// k-points per CTA, the reflectors one at a time; no reductions across threads.  (A CTA per k-point
// keeps 4 W lanes, one warp at W = 6, and pays its barriers for 4 reflectors.)
template <int WM>
__global__ void __launch_bounds__(256) reflect_small_kernel(int W, int n, int kpc, EighBufs b,
                                                            const double* __restrict__ Z,
                                                            double2* __restrict__ Uout) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int4* swA = reinterpret_cast<int4*>(smraw);   // [kpc][W][W]: column j = unit reflector w_j
  const int t = threadIdx.x;
  const int lk = t / W, c = t - lk * W;
  const int64_t k = (int64_t)blockIdx.x * kpc + lk;
  const bool live = lk < kpc && k < n;
  int4* sw = swA + (size_t)lk * W * W;
  if (live) {   // thread c stages row c
    const double2* R = b.refl + (size_t)k * W * W + (size_t)c * W;
    for (int j = 0; j < W - 2; ++j) {
      int4 w = make_int4(0, 0, 0, 0);
      if (c > j) {
        const double f = sqrt(0.5 * b.tau[k * W + j]);
        const double2 v = R[j];
        w = fx::climbs(fx::from_double(v.x * f, 58), fx::from_double(v.y * f, 58));
      }
      sw[c * W + j] = w;
    }
  }
  __syncthreads();
  if (!live) return;
  int4 u[WM];
  bool bad = false;   // an infinite or NaN entry of Z
#pragma unroll
  for (int r = 0; r < WM; ++r) {
    u[r] = make_int4(0, 0, 0, 0);
    if (r < W) {
      const double z = Z[(size_t)k * W * W + (size_t)r * W + c];
      bad |= !fx::finite(z);
      const double2 p = b.phase[k * W + r];
      u[r] = fx::climbs(fx::from_double(p.x * z, 58), fx::from_double(p.y * z, 58));
    }
  }
#pragma unroll 1
  for (int j = W - 3; j >= 0; --j) {
    fx::Acc s;
    fx::zero(s);
#pragma unroll
    for (int r = 1; r < WM; ++r)
      if (r < W && r > j) {
        const int4 w = sw[r * W + j];
        fx::cmadc(s, w, -w.z, -w.w, u[r]);
      }
    // h = w^dagger u (units 2^-60), u -= 2 w h
    const int4 h = fx::climbs(fx::fold_shift(s.rh, s.rm, 2), fx::fold_shift(s.ih, s.im, 2));
#pragma unroll
    for (int r = 1; r < WM; ++r)
      if (r < W && r > j) {
        const int4 w = sw[r * W + j];
        fx::Acc d;
        fx::zero(d);
        fx::cmad(d, w, -w.z, -w.w, fx::pin(h));
        u[r] = fx::climbs(fx::value(u[r].x, u[r].y) - fx::fold_shift(d.rh, d.rm, 1),
                          fx::value(u[r].z, u[r].w) - fx::fold_shift(d.ih, d.im, 1));
      }
  }
  double2* Uk = Uout + (size_t)k * W * W;
#pragma unroll
  for (int r = 0; r < WM; ++r)
    if (r < W) {
      double2 v = make_double2(fx::to_double(fx::value(u[r].x, u[r].y), -58),
                               fx::to_double(fx::value(u[r].z, u[r].w), -58));
      if (bad) v.x = v.y = __longlong_as_double(0x7FF8000000000000ll);
      Uk[r * W + c] = v;
    }
}

}  // namespace

cudaError_t launch_unorm(const double2* U, int W, int n, int* ue, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  unorm_kernel<<<n, 256, 0, s>>>(U, W, ue);
  return cudaGetLastError();
}

cudaError_t launch_berry_fix(const double* E, const double2* U, const double* Xp, const double* Yp,
                             int64_t ld, int W, int n, const double* etas, int n_eta, double* Om,
                             int64_t eta_stride, const int* ue, cudaStream_t s, int pad) {
  if (n <= 0) return cudaSuccess;
  if (W > 64 || n_eta > MAXE) return cudaErrorInvalidValue;
  // Output tile of a thread: 4 x 2 from W = 13 (two 16-byte operand loads fewer per product than 2 x 2),
  // 2 x 2 below, where 4 x 2 leaves more of the tile outside the matrix.  The threads per k-point
  // cover W exactly up to that granularity, so an uneven W wastes no products on padding to 16 or 64.
  // Few matrices of the caller's: one output per thread and one matrix per CTA, BERRY_FEW
  const bool few = ue != nullptr && W <= 16 && n <= BERRY_FEW;
  const bool small = W < 13;
  const int TM = few ? 1 : small ? 2 : 4, TN = few ? 1 : 2;
  // skipped pairs assume NX TN = NY TM: the common span is W rounded up to 4 (2 when small)
  const int span = (W + TM - 1) / TM * TM;
  const int NY = span / TM, NX = span / TN;
  const int nthr = NX * NY;
  const int KPC = few ? 1 : std::max(1, 256 / nthr);
  const int block = (KPC * nthr + 31) / 32 * 32;
  const int LD = pad ? W | 1 : W;   // pad = 0: the padding ablation
  const size_t sm = (size_t)KPC * W * LD * 2 * sizeof(int4) + (size_t)TM * TN * block * sizeof(double2) +
                    (size_t)KPC * W * sizeof(double) + (size_t)KPC * 24;
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(n + KPC - 1) / KPC, block, sm, s>>>(E, U, Xp, Yp, ld, W, n, etas, n_eta, Om, eta_stride, NX,
                                                NY, KPC, LD, ue);
    return cudaGetLastError();
  };
  if (few) return go(berry_fix_kernel<1, 1>);
  return small ? go(berry_fix_kernel<2, 2>) : go(berry_fix_kernel<4, 2>);
}

cudaError_t launch_reflect_fix(int W, int n, EighBufs b, const double* Z, double2* U, cudaStream_t s,
                               int pad) {
  if (n <= 0) return cudaSuccess;
  if (W > LARGE_W_MAX) return cudaErrorInvalidValue;
  if (W <= 16) {
    const int kpc = 256 / W;
    const size_t sm = (size_t)kpc * W * W * sizeof(int4);
    auto go = [&](auto kern) -> cudaError_t {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e != cudaSuccess) return e;
      kern<<<(n + kpc - 1) / kpc, 256, sm, s>>>(W, n, kpc, b, Z, U);
      return cudaGetLastError();
    };
    return W <= 8 ? go(reflect_small_kernel<8>) : go(reflect_small_kernel<16>);
  }
  // all columns up to W = 64, half of them above (W = 97, 2,736 k-points: halves 6.7 ms, thirds 7.3, quarters
  // 6.9; W = 128: 14.5, 14.7, 15.8; W = 64, 4,096: all columns 2.55, halves 2.65; W = 32: 0.46, 0.50)
  const int nb = W <= 64 ? 1 : 2, CB = (W + nb - 1) / nb;
  const int LD = pad ? CB | 1 : CB;
  const size_t sm = ((size_t)W * LD + 2 * (size_t)W * RF_NB + 12 + W) * sizeof(int4) + (size_t)W * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(reflect_fix_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int nt = std::min(RF_NT, (4 * CB + 31) / 32 * 32);   // four lanes per column
  reflect_fix_kernel<<<dim3(n, (W + CB - 1) / CB), nt, sm, s>>>(W, b, Z, U, CB, LD);
  return cudaGetLastError();
}

}  // namespace kubo
