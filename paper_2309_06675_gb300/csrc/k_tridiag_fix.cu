// Householder reduction H = Q D T D^dagger Q^dagger in FP64 grade on the integer pipe (fixed.cuh), for
// the FP64 mode (the mixed modes' reduction stays the FP64 one of k_eigh.cu).
//
// The FP64 reduction runs at 92 % of the FP64 pipe (8 multiply-adds of 16 clocks per warp
// for each trailing element and column).  Here the trailing matrix is held as 59-bit fixed-point
// numbers relative to a power of two above its Frobenius norm, which the reduction's unitary
// similarities never exceed; its symmetric product and its rank-2 update are sums of fixed-point
// products.  A rounding is 2^-60 of that norm, at most 2^-57 of the spectral norm at W = 64, where an
// FP64 update rounds every entry to 2^-54 of itself several times.  (Each is rounded once, to the nearest: see
// fold_shift() for what a bias costs.  Against an 80-bit reference, geometric means over 144 k-points of random models, FP64
// reduction -> this one: largest error of a k-point's eigenvalues 1.4e-15 -> 5.7e-16 of the norm at W = 64, 2.3e-15 -> 7.5e-16
// at 128; of its curvatures 8.0e-14 -> 3.6e-14 and 2.4e-13 -> 1.4e-13 of the largest.)  Only what one warp does per
// column (the column's norm, the Householder vector's scale) is FP64.
//
// Uncoupled blocks (consecutive orbitals without a matrix element to the others: layers, spins) whose rows' largest
// entries differ by 2^4 or more have a scale each, so that a small block keeps its own relative accuracy beside a
// large one: a reflector never leaves its block.
//
// KP k-points per CTA, TPK threads each (2 x 128 at W <= 64, 4 x 64 at 32, 8 x 32 at 16, 16 x 16 at 8,
// 1 x 256 or 384 above 64); warp 0 runs the scalar steps of all KP k-points at once, 32 / KP lanes each.
// Per column i with reflector I - 2 w w^dagger (w a unit vector, kept in column i of A):
//   1 (all)     partial sums of p = A w
//   2 (warp 0)  p, K = w^dagger p, h = p - K w
//   3 (warp 0)  column i + 1 of A <- A - 2 (w h^dagger + h w^dagger), its |x|, and the next
//               w = v / |v|, v = x + e^{i arg x_0} |x| e_0
//     (others)  the rest of the lower triangle of that update
// The next column's reflector is a chain of some 2,000 clocks; beside the update it is hidden (on
// its own between two barriers: W = 64, 4,096 k-points 2.87 ms, beside it 2.77; W = 97, 2,744, with one CTA per SM: 11.4
// and 11.0, and 6.5 with the two CTAs of launch_tridiag_fix).
// What bounds it: the integer multiply-adds (12 per complex product) and, for short columns, the
// latency of step 2, which the other CTAs of the SM fill.
#include <algorithm>

#include "fixed.cuh"
#include "kubo_internal.cuh"

namespace kubo {

namespace {

__device__ __forceinline__ int tri(int r, int c) { return (r * (r + 1) >> 1) + c; }

__host__ __device__ constexpr int sp_len(int W, int TPK) { return TPK > 2 * W ? TPK : 2 * W; }
__host__ __device__ constexpr size_t fix_bytes_per_k(int W, int TPK) {
  return ((size_t)W * (W + 1) / 2 + sp_len(W, TPK) + W) * 16;
}

// 2^e above the Frobenius norm: |entries|^2 add up to at most sq 2^(2 (emax - 1037))
__device__ __forceinline__ int norm_exp(int emax, unsigned long long sq) {
  return sq == 0ull ? 0 : emax - 1037 + ((64 - __clzll((long long)sq) + 1) >> 1);
}
// an entry's part of that sum: hx, hy the upper halves of its parts' magnitudes (m + 1 above the 15 leading
// bits at exponent emax)
__device__ __forceinline__ unsigned long long norm_part(unsigned hx, unsigned hy, int emax) {
  const int sx = emax - (int)(hx >> 20), sy = emax - (int)(hy >> 20);
  const unsigned m = (hx && sx < 15 ? (((hx & 0xFFFFFu) | 0x100000u) >> 6) >> sx : 0u) + 1u;
  const unsigned l = (hy && sy < 15 ? (((hy & 0xFFFFFu) | 0x100000u) >> 6) >> sy : 0u) + 1u;
  return 2ull * ((hx ? m * m : 0u) + (unsigned long long)(hy ? l * l : 0u));   // (diagonal: twice its share)
}
__device__ __forceinline__ unsigned upper_mag(double x) { return (unsigned)(mag_bits(x) >> 32); }

constexpr int SPLIT_SPREAD = 4;   // binary orders between rows from which uncoupled blocks have their own scale

template <int KP, int TPK, int MINB>
__global__ void __launch_bounds__(KP* TPK, MINB)
    tridiag_fix_kernel(const double* __restrict__ Hp, int64_t ld, int W, int n, EighBufs b) {
  constexpr int LPK = 32 / KP;   // warp 0's lanes per k-point; four rows each cover W
  extern __shared__ __align__(16) unsigned char smraw[];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int g = t / TPK, th = t - g * TPK;
  const int NA = W * (W + 1) / 2, SP = sp_len(W, TPK);
  const size_t per_k = (size_t)NA + SP + W;
  int4* base = reinterpret_cast<int4*>(smraw);
  int4* A = base + g * per_k;                                       // lower triangle, packed by rows
  longlong2* sp = reinterpret_cast<longlong2*>(A + NA);             // partial sums; then h | w as limbs
  unsigned char* rowtab = smraw + KP * per_k * 16;                  // row of a strictly lower element
  __shared__ unsigned long long s_sq[KP];
  __shared__ unsigned s_max[KP];
  __shared__ int s_act[2][KP];   // of the odd and of the even columns
  __shared__ int s_lo[KP];       // exponent of the smallest row; from then on: blocks have their own scale
  const int64_t k = (int64_t)blockIdx.x * KP + g;
  const bool live = k < n;

  if (t < KP) { s_sq[t] = 0ull; s_max[t] = 0u; s_lo[t] = 0; }
  int open = 0;   // an element beside the diagonal is zero
  for (int r = 1 + warp; r < W; r += KP * TPK / 32)
    for (int c = lane; c < r; c += 32) rowtab[r * (r - 1) / 2 + c] = (unsigned char)r;
  __syncthreads();
  // ---- load, scale: 2^e above the Frobenius norm (|entry| < (m + 1) 2^(emax - 1037), m its 15 leading
  // bits at the largest exponent)
  {
    double2* Ad = reinterpret_cast<double2*>(A);
    const double* P = Hp + (live ? k : 0) * ld;
    unsigned mx = 0u;
    if (live)
      for (int idx = th; idx < NA; idx += TPK) {
        int r = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
        while (tri(r, 0) > idx) --r;
        while (tri(r + 1, 0) <= idx) ++r;
        const int c = idx - tri(r, 0);
        const double2 a = r == c ? make_double2(P[r * W + r], 0.0) : make_double2(P[c * W + r], -P[r * W + c]);
        Ad[idx] = a;
        mx = max(mx, (unsigned)(max(mag_bits(a.x), mag_bits(a.y)) >> 32));
      }
    if (mx) atomicMax(&s_max[g], mx);
    __syncthreads();
    const int emax = (int)(s_max[g] >> 20);
    unsigned long long s = 0ull;
    if (live) {
      for (int idx = th; idx < NA; idx += TPK) {
        const double2 a = Ad[idx];
        s += norm_part(upper_mag(a.x), upper_mag(a.y), emax);
      }
      for (int r = 1 + th; r < W; r += TPK) {
        const double2 a = Ad[tri(r, r - 1)];
        open |= (mag_bits(a.x) | mag_bits(a.y)) == 0ull;
      }
    }
    if (s) atomicAdd(&s_sq[g], s);
    open = __syncthreads_or(open);
  }
  const int emax = (int)(s_max[g] >> 20);
  const bool bad = emax == 0x7FF;
  const int e = bad ? 0 : norm_exp(emax, s_sq[g]);
  if (open) {   // (the same for the CTA)
    // a thread per row, tables in the place of the partial sums: the first column with an entry, the first row
    // of the row's block, that block's largest entry and sum of squares
    unsigned long long* bsq = reinterpret_cast<unsigned long long*>(sp);
    int* first = reinterpret_cast<int*>(bsq + W);
    unsigned* bmax = reinterpret_cast<unsigned*>(first + W);
    int* start = reinterpret_cast<int*>(bmax + W);
    const double2* Ad = reinterpret_cast<const double2*>(A);
    const bool row = live && !bad && th < W;   // (W <= TPK for every instance)
    unsigned rowmax = 0u;
    if (th == 0) s_lo[g] = 0x7FF;
    __syncthreads();
    if (row) {
      int f = th;
      for (int c = th; c >= 0; --c) {
        const double2 a = Ad[tri(th, c)];
        if ((mag_bits(a.x) | mag_bits(a.y)) != 0ull) f = c;
        rowmax = max(rowmax, max(upper_mag(a.x), upper_mag(a.y)));
      }
      for (int i = th + 1; i < W; ++i) {
        const double2 a = Ad[tri(i, th)];
        rowmax = max(rowmax, max(upper_mag(a.x), upper_mag(a.y)));
      }
      first[th] = f;
      bmax[th] = 0u;
      bsq[th] = 0ull;
      if (rowmax >> 20) atomicMin(&s_lo[g], (int)(rowmax >> 20));
    }
    __syncthreads();
    const bool apart = live && !bad && emax - s_lo[g] >= SPLIT_SPREAD;
    if (__syncthreads_or(apart)) {
      const bool mine = apart && row;
      if (mine) {   // the last row up to this one from which on no row reaches in front of it
        int m = W, b0 = 0;
        for (int i = W - 1; i > 0; --i) {
          m = min(m, first[i]);
          if (i <= th && m >= i) { b0 = i; break; }
        }
        start[th] = b0;
        atomicMax(&bmax[b0], rowmax >> 20);
      }
      __syncthreads();
      if (mine) {
        const int b0 = start[th], em = (int)bmax[b0];
        unsigned long long s = 0ull;
        for (int c = b0; c <= th; ++c) {
          const double2 a = Ad[tri(th, c)];
          s += norm_part(upper_mag(a.x), upper_mag(a.y), em);
        }
        atomicAdd(&bsq[b0], s);
      }
      __syncthreads();
      // the rows' exponents, kept in lam until the outputs are scaled back
      if (mine) b.lam[k * W + th] = (double)norm_exp((int)bmax[start[th]], bsq[start[th]]);
    }
    if (th == 0) s_lo[g] = apart ? 1 : 0;
    __syncthreads();
  }
  const bool split = s_lo[g] != 0;
  if (live) {
    const double2* Ad = reinterpret_cast<const double2*>(A);
    for (int idx = th; idx < NA; idx += TPK) {
      const double2 a = Ad[idx];
      int ea = e;
      if (split) {
        int r = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
        while (tri(r, 0) > idx) --r;
        while (tri(r + 1, 0) <= idx) ++r;
        ea = (int)b.lam[k * W + r];
      }
      A[idx] = bad ? make_int4(0, 0, 0, 0)
                   : fx::climbs(fx::from_double(a.x, fx::BITS - ea), fx::from_double(a.y, fx::BITS - ea));
    }
  }
  __syncthreads();

  // warp 0's k-point
  const int kk = lane / LPK, l = lane - kk * LPK;
  int4* Ak = base + kk * per_k;
  longlong2* spk = reinterpret_cast<longlong2*>(Ak + NA);
  double2* betak = reinterpret_cast<double2*>(spk + SP);   // beta_i, in units of 2^(e - 59)
  const int64_t kw = (int64_t)blockIdx.x * KP + kk;
  const bool livek = kw < n;

  // warp 0, for its k-point: the reflector of column i (rows i + 1 + r).  upd: the previous step's
  // rank-2 update of that column (its trailing column 0) is still to be made, from h and w in spk.
  auto reflector = [&](int i, bool upd) {
    const int o = i + 1, m = W - 1 - i;
    double xr[4], xi[4];
    double s2 = 0.0;
    const int4* h4 = reinterpret_cast<const int4*>(spk);
    const int4 h0 = upd ? h4[0] : make_int4(0, 0, 0, 0), w0 = upd ? h4[W] : h0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = l + LPK * q;
      xr[q] = xi[q] = 0.0;
      if (r < m && livek) {
        int4* pa = &Ak[tri(o + r, i)];
        const int4 a = *pa;
        long long vx = fx::value(a.x, a.y), vy = fx::value(a.z, a.w);
        if (upd) {   // row r here is row r + 1 of the previous trailing block
          const int4 hr = h4[r + 1], wr = h4[W + r + 1];
          fx::Acc acc;
          fx::zero(acc);
          const int4 hp = fx::pin(h0), wp = fx::pin(w0);
          fx::cmadc(acc, hp, -hp.z, -hp.w, wr);   // w_r conj(h_0) + h_r conj(w_0), units 2^-61
          fx::cmadc(acc, wp, -wp.z, -wp.w, hr);
          vx -= fx::fold_shift(acc.rh, acc.rm, 1);
          vy -= fx::fold_shift(acc.ih, acc.im, 1);
          *pa = fx::climbs(vx, vy);
        }
        xr[q] = (double)vx;
        xi[q] = (double)vy;
        if (r > 0) s2 = fma(xr[q], xr[q], fma(xi[q], xi[q], s2));
      }
    }
    if (upd && l == 0 && livek) {   // the diagonal entry above the column
      int4* pa = &Ak[tri(i, i)];
      long long hh = 0, c = 0;
      fx::mad(hh, h0.x, w0.x); fx::mad(c, h0.x, w0.y); fx::mad(c, h0.y, w0.x);
      fx::mad(hh, h0.z, w0.z); fx::mad(c, h0.z, w0.w); fx::mad(c, h0.w, w0.z);
      const int2 x = fx::limbs(fx::value(pa->x, pa->y) - fx::fold(hh, c));
      *pa = make_int4(x.x, x.y, 0, 0);
    }
    if (i >= W - 2) return;   // (the last column is only brought up to date)
#pragma unroll
    for (int f = LPK / 2; f > 0; f >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, f);
    const double ax = __shfl_sync(0xffffffffu, xr[0], kk * LPK), ay = __shfl_sync(0xffffffffu, xi[0], kk * LPK);
    // |x| in the even lanes, |x_0| in the odd ones: one reciprocal square root
    const double aa2 = fma(ax, ax, ay * ay);
    const double arg = (l & 1) ? aa2 : aa2 + s2;
    const double ri = mag_bits(arg) != 0ull ? rsqrt(arg) : 0.0;
    const double root = arg * ri;
    const double nrm = __shfl_sync(0xffffffffu, root, kk * LPK);
    const double aa = __shfl_sync(0xffffffffu, root, kk * LPK + 1);
    const double ra = __shfl_sync(0xffffffffu, ri, kk * LPK + 1);
    const bool az = mag_bits(aa2) == 0ull;
    const double px = az ? 1.0 : ax * ra, py = az ? 0.0 : ay * ra;   // the unit phase of x_0
    const bool act = mag_bits(s2) != 0ull;
    if (act) {
      // v = (ph (|x| + |x_0|), x_1, ...), |v|^2 = 2 |x| (|x| + |x_0|)
      const double tt = nrm + aa;
      const double f = rsqrt(2.0 * nrm * tt);
      if (l == 0) {
        xr[0] = px * tt;
        xi[0] = py * tt;
        betak[i] = make_double2(-px * nrm, -py * nrm);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = l + LPK * q;
        if (r < m)
          Ak[tri(o + r, i)] = fx::climbs(fx::from_double(xr[q] * f, 58), fx::from_double(xi[q] * f, 58));
      }
    } else if (l == 0 && livek) {
      betak[i] = make_double2(ax, ay);   // no reflection
    }
    if (l == 0) {
      s_act[i & 1][kk] = act ? 1 : 0;
      if (livek) b.tau[kw * W + i] = act ? 2.0 : 0.0;
    }
  };

  if (warp == 0 && W > 2) reflector(0, false);
  __syncthreads();
  for (int i = 0; i < W - 2; ++i) {
    const int o = i + 1;       // first row of the trailing block
    const int m = W - 1 - i;   // its size
    const int P = max(1, min(TPK / m, 8));   // column partitions of a row
    if (s_act[i & 1][g]) {
      const int part = th / m, r = th - part * m;
      if (part < P) {
        fx::Acc acc;
        fx::zero(acc);
        const int rowb = tri(o + r, o);
        for (int c = part; c < m; c += P) {
          const bool up = c > r;   // mirrored: the conjugate of (c, r)
          const int4 a = A[up ? tri(o + c, o + r) : rowb + c];
          const int4 w = A[tri(o + c, i)];
          const int nz = -a.z, nw = -a.w;
          const int4 as = make_int4(a.x, a.y, up ? nz : a.z, up ? nw : a.w);
          fx::cmad(acc, as, up ? a.z : nz, up ? a.w : nw, w);
        }
        sp[part * m + r] = make_longlong2(fx::fold(acc.rh, acc.rm), fx::fold(acc.ih, acc.im));
      }
    }
    __syncthreads();
    if (warp == 0 && s_act[i & 1][kk]) {
      // (a k-point's lanes take this together; the shuffles stay inside its group)
      const unsigned gm = (LPK == 32 ? 0xffffffffu : ((1u << (LPK & 31)) - 1u)) << (kk * LPK);
      long long pr[4], pi[4];
      int4 w[4];
      long long ks = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = l + LPK * q;
        pr[q] = pi[q] = 0;
        w[q] = make_int4(0, 0, 0, 0);
        if (r < m) {
          long long sx = 0, sy = 0;
          for (int p = 0; p < P; ++p) {
            const longlong2 v = spk[p * m + r];
            sx += v.x;
            sy += v.y;
          }
          pr[q] = fx::rshift(sx, 2);
          pi[q] = fx::rshift(sy, 2);
          w[q] = Ak[tri(o + r, i)];
          const int4 p4 = fx::climbs(pr[q], pi[q]);
          long long h = 0, c = 0;   // Re(conj(w) p)
          fx::mad(h, w[q].x, p4.x); fx::mad(c, w[q].x, p4.y); fx::mad(c, w[q].y, p4.x);
          fx::mad(h, w[q].z, p4.z); fx::mad(c, w[q].z, p4.w); fx::mad(c, w[q].w, p4.z);
          ks += fx::fold(h, c);
        }
      }
#pragma unroll
      for (int f = LPK / 2; f > 0; f >>= 1) ks += __shfl_xor_sync(gm, ks, f);
      const int2 K = fx::limbs(fx::rshift(ks, 2));
      __syncwarp(gm);   // every partial sum of the k-point has been read
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = l + LPK * q;
        if (r < m) {
          long long rh = 0, rm = 0, ih = 0, im = 0;
          const int4 wq = fx::pin(w[q]), Kp = fx::pin(make_int4(K.x, K.y, 0, 0));
          fx::mad(rh, Kp.x, wq.x); fx::mad(rm, Kp.x, wq.y); fx::mad(rm, Kp.y, wq.x);
          fx::mad(ih, Kp.x, wq.z); fx::mad(im, Kp.x, wq.w); fx::mad(im, Kp.y, wq.z);
          int4* s4 = reinterpret_cast<int4*>(spk);
          s4[r] = fx::climbs(pr[q] - fx::fold_shift(rh, rm, 2), pi[q] - fx::fold_shift(ih, im, 2));
          s4[W + r] = w[q];
        }
      }
    }
    __syncthreads();
    // Warp 0 brings the next column up to date and forms its reflector (a chain of some 2,000 clocks)
    // while the other warps update the rest of all KP trailing blocks.
    if (warp == 0) {
      reflector(i + 1, s_act[i & 1][kk] != 0);
    } else {
      const int m1 = m - 1;                  // trailing rows and columns 1 .. m - 1
      const int nl = m1 * (m1 + 1) / 2;      // their lower triangle with the diagonal
      const FastDiv dn((uint32_t)nl);
      for (int it = t - 32; it < KP * nl; it += KP * TPK - 32) {
        const int gg = KP == 1 ? 0 : (int)dn.div(it), idx = it - gg * nl;
        if (!s_act[i & 1][gg]) continue;
        // packed with its diagonal: row r' >= c', from the table of strictly lower elements of the block
        // one larger (row r' + 1, column c')
        const int r = rowtab[idx], c = idx - r * (r - 1) / 2 + 1;
        int4* Ag = base + gg * per_k;
        const int4* hb = Ag + NA;
        const int4* wb = hb + W;
        const int4 hc = hb[c], wr = wb[r], wc = wb[c], hr = hb[r];
        fx::Acc acc;
        fx::zero(acc);
        fx::cmadc(acc, hc, -hc.z, -hc.w, wr);   // w_r conj(h_c) + h_r conj(w_c), units 2^-61
        fx::cmadc(acc, wc, -wc.z, -wc.w, hr);
        int4* pa = &Ag[tri(o + r, o + c)];
        const int4 a = *pa;
        *pa = fx::climbs(fx::value(a.x, a.y) - fx::fold_shift(acc.rh, acc.rm, 1),
                         fx::value(a.z, a.w) - fx::fold_shift(acc.ih, acc.im, 1));
      }
    }
    __syncthreads();
  }

  // ---- outputs
  const double nan = __longlong_as_double(0x7FF8000000000000ll);
  if (live) {
    double* dout = b.d + k * W;
    for (int j = th; j < W; j += TPK) {
      const int4 a = A[tri(j, j)];
      const int ea = split ? (int)b.lam[k * W + j] : e;
      dout[j] = bad ? nan : fx::scale_pow2((double)fx::value(a.x, a.y), ea - fx::BITS);
      if (j >= W - 2) b.tau[k * W + j] = 0.0;
    }
    double2* rout = b.refl + (size_t)k * W * W;
    const FastDiv dW(W);
    for (int idx = th; idx < W * W; idx += TPK) {
      const int r = (int)dW.div(idx), c = idx - r * W;
      double2 v = make_double2(0.0, 0.0);
      if (r > c && c < W - 2) {
        const int4 a = A[tri(r, c)];
        v = make_double2(fx::to_double(fx::value(a.x, a.y), -58), fx::to_double(fx::value(a.z, a.w), -58));
      }
      rout[idx] = v;
    }
  }
  if (warp == 0) {
    // |beta_j|, and the phases D_0 = 1, D_{j+1} = D_j beta_j / |beta_j| as a scan over the k-point's lanes,
    // lane l with j = 4 l .. 4 l + 3
    const int emk = (int)(s_max[kk] >> 20);
    const unsigned long long sqk = s_sq[kk];
    const bool badk = emk == 0x7FF;
    const int ek = badk ? 0 : norm_exp(emk, sqk);
    const bool splitk = s_lo[kk] != 0;
    double2 u[4], pr = make_double2(1.0, 0.0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = 4 * l + q;
      u[q] = make_double2(1.0, 0.0);
      if (j + 1 < W && livek) {
        double2 bj;
        if (j == W - 2) {
          const int4 a = Ak[tri(W - 1, W - 2)];
          bj = make_double2((double)fx::value(a.x, a.y), (double)fx::value(a.z, a.w));
        } else {
          bj = betak[j];
        }
        const double a2 = fma(bj.x, bj.x, bj.y * bj.y);
        double a = 0.0;
        if (mag_bits(a2) != 0ull) {
          const double ra = rsqrt(a2);
          a = a2 * ra;
          u[q] = make_double2(bj.x * ra, bj.y * ra);
        }
        // (an infinite or NaN entry: T = NaN I, which the QL iteration leaves as it is)
        const int ea = splitk ? (int)b.lam[kw * W + j] : ek;
        b.e[kw * W + j] = badk ? 0.0 : fx::scale_pow2(a, ea - fx::BITS);
      }
      pr = cmul(pr, u[q]);
    }
    double2 sc = pr;
#pragma unroll
    for (int off = 1; off < LPK; off <<= 1) {
      double2 o2;
      o2.x = __shfl_up_sync(0xffffffffu, sc.x, off, LPK);
      o2.y = __shfl_up_sync(0xffffffffu, sc.y, off, LPK);
      if (l >= off) sc = cmul(o2, sc);
    }
    double2 D;
    D.x = __shfl_up_sync(0xffffffffu, sc.x, 1, LPK);
    D.y = __shfl_up_sync(0xffffffffu, sc.y, 1, LPK);
    if (l == 0) D = make_double2(1.0, 0.0);
    if (livek) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = 4 * l + q;
        if (j < W) b.phase[kw * W + j] = D;
        D = cmul(D, u[q]);
      }
      if (l == 0) b.e[kw * W + W - 1] = 0.0;
    }
  }
}

}  // namespace

cudaError_t launch_tridiag_fix(const double* Hp, int64_t ld, int W, int n, EighBufs b, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  auto go = [&](auto kern, int KP, int TPK) -> cudaError_t {
    const size_t sm = KP * fix_bytes_per_k(W, TPK) + (size_t)W * (W - 1) / 2;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(n + KP - 1) / KP, KP * TPK, sm, s>>>(Hp, ld, W, n, b);
    return cudaGetLastError();
  };
  if (W <= 8) return go(tridiag_fix_kernel<16, 16, 3>, 16, 16);
  if (W <= 16) return go(tridiag_fix_kernel<8, 32, 3>, 8, 32);
  if (W <= 32) return go(tridiag_fix_kernel<4, 64, 3>, 4, 64);
  if (W <= 64) return go(tridiag_fix_kernel<2, 128, 3>, 2, 128);
  // above 64 one k-point per CTA, and more CTAs per SM before more threads: three of 256 threads where their
  // shared memory fits (W <= 90), else 384 (two CTAs to W = 108).  4,096 k-points: W = 66 3.5 ms, W = 80 5.1
  // (one CTA of 512: 8.6, 11.6; two of 512: 5.0, 6.9); 2,744: W = 97 6.5, W = 107 8.0, W = 128 17.5
  // (256 threads: 6.7, 8.4, 19.2; one of 512: 11.0, 13.2, 18.2).
  if (3 * (fix_bytes_per_k(W, 256) + (size_t)W * (W - 1) / 2 + 1024 + 64) <= (size_t)228 * 1024)
    return go(tridiag_fix_kernel<1, 256, 3>, 1, 256);
  return go(tridiag_fix_kernel<1, 384, 2>, 1, 384);
}

}  // namespace kubo
