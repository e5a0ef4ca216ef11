// Batched complex W x W products of FP64 grade on the 5th-generation tensor cores, W <= 128, and
// the curvature of Eq. 3 from the velocity matrices they form.
//
//   C[k] = op(A[k]) op(B[k]) (+ C[k]),  op: identity, conjugate transpose, or (A) a Hermitian matrix
//   from its packed real row
//
// Every real and imaginary part is cut into seven signed base-256 digits relative to its matrix's
// largest entry (digits.cuh) and the digit products of the levels i + j <= 7 are kept (34 of 49, level
// 7 without the single pair that needs an eighth digit): the operands' rounding, 2^-56 of the largest
// entries, is the error that remains (levels 8 and beyond are 2^-65 per product).  A level sum over 128 of
// K is an integer of at most 7 x 128 x 2^14 < 2^24, exact in the FP32 accumulator.
//
// One tile is 64 complex rows by up to 64 columns as a real product [re; im] (M = 128) with K = 2 W:
// the rows [Ar | -Ai] and [Ai | Ar] against [Br; Bi].  A chunk is 16 of the inner index (32 of K); the
// staging warps load it in FP64, cut it and write it to shared memory (128-byte swizzle, a row of 64
// BF16 holding two chunks) while the MMAs of the other half run; the eight level sums of a
// tile fill the 512 TMEM columns (N = 64); eight warps add them in one int64 (units
// 2^-55 of the operand scales) and convert with integer instructions: FP64 conversions would take longer
// than the products (the FP64 pipe converts 2 lanes per clock).
//
// What bounds it: the MMAs (34 x 128 x N x 2 W / 4096 clocks per tile) and the staging of the next chunk
// (about 500 instructions for each 8 complex entries) take about the same time.  FP64 FMA kernels
// of the same products ran at 1.1 TFLOP/s; measured here: see the table beside the launcher.
//
// Every mbarrier wait is bounded; a wait that gives up sets ST_TIMEOUT and the CTA returns.
#include <algorithm>

#include <cuda_bf16.h>

#include "digits.cuh"
#include "fixed.cuh"
#include "kubo_internal.cuh"
#include "tc_ptx.cuh"

namespace kubo {

namespace {

using namespace tc;
using namespace dig;

constexpr int BM = 128;             // [re; im] of 64 complex rows
constexpr int CH = 16;              // inner indices per chunk (K = 32)
constexpr int GROUP = 4;            // chunks per drain (K = 128)
constexpr int NLEV = 8;
constexpr int ROW_BYTES = 128;      // 64 BF16: two chunks
constexpr int A_SLICE = BM * ROW_BYTES;          // 16 KB
constexpr int STAGE_THREADS = 256;
constexpr int EPI_THREADS = 256;
constexpr int THREADS = STAGE_THREADS + EPI_THREADS;   // 16 warps: 128 registers each
constexpr int TMEM_COLS = 512;
constexpr int E_MIN = -1080;        // exponent of an all-zero operand

__host__ __device__ __forceinline__ uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ int op_exp(const ZOp& o, int64_t k) { return o.e ? max(o.e[k], E_MIN) : 0; }

// v 2^e in FP64 (v = 0 or rounded half up of the magnitude), by integer instructions
__device__ __forceinline__ double int_to_double(long long v, int e) {
  const long long s = v >> 63;
  const unsigned long long a = (unsigned long long)((v ^ s) - s);
  if (a == 0ull) return 0.0;
  const int lz = __clzll((long long)a);
  const int ex = 1023 + 63 - lz + e;
  if (ex < 1 || ex > 2045) return fx::scale_pow2((double)v, e);
  const unsigned long long m = (((a << lz) >> 10) + 1ull) >> 1;   // 2^52 .. 2^53
  return __longlong_as_double((long long)((((unsigned long long)(ex - 1) << 52) + m) |
                                          ((unsigned long long)s & 0x8000000000000000ull)));
}

// 8 complex entries of a chunk: rows r (A) or columns r (B), inner indices q0 .. q0 + 7, zeros outside
// the matrix
template <int KIND>
__device__ __forceinline__ void load8(const ZOp& o, int64_t k, int W, bool is_b, int r, int q0,
                                      double2 (&v)[8]) {
  if (KIND == 2) {
    const double* P = reinterpret_cast<const double*>(o.p) + k * o.ld;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int q = q0 + i;
      v[i] = make_double2(0.0, 0.0);
      if (r < W && q < W) {
        const double a = P[r * W + q], b = P[q * W + r];
        v[i] = r < q ? make_double2(a, b) : r > q ? make_double2(b, -a) : make_double2(a, 0.0);
      }
    }
  } else {
    const double2* P = reinterpret_cast<const double2*>(o.p) + k * (int64_t)W * W;
    // A: (r, q) of the matrix or, conjugated, (q, r); B: (q, r) or, conjugated, (r, q)
    const bool row = (KIND == 0) != is_b;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int q = q0 + i;
      v[i] = make_double2(0.0, 0.0);
      if (r < W && q < W) {
        v[i] = row ? P[r * W + q] : P[q * W + r];
        if (KIND == 1) v[i].y = -v[i].y;
      }
    }
  }
}

// the seven digit slices of 8 values at 16-byte unit u of a row (and, for A, of a second row)
__device__ __forceinline__ void put8(const uint32_t (&d)[8][ND], unsigned char* row, int sw,
                                     int slice_bytes, int u) {
#pragma unroll
  for (int s = 0; s < ND; ++s) {
    uint4 w;
    w.x = bf16_pair(d[0][s], d[1][s]);
    w.y = bf16_pair(d[2][s], d[3][s]);
    w.z = bf16_pair(d[4][s], d[5][s]);
    w.w = bf16_pair(d[6][s], d[7][s]);
    *reinterpret_cast<uint4*>(row + s * slice_bytes + ((u ^ sw) << 4)) = w;
  }
}
// the same digits to two rows, the second with the opposite sign
__device__ __forceinline__ void put8_pm(const uint32_t (&d)[8][ND], unsigned char* row, int u,
                                        unsigned char* nrow, int nu, int sw, int slice_bytes) {
#pragma unroll
  for (int s = 0; s < ND; ++s) {
    uint4 w;
    w.x = bf16_pair(d[0][s], d[1][s]);
    w.y = bf16_pair(d[2][s], d[3][s]);
    w.z = bf16_pair(d[4][s], d[5][s]);
    w.w = bf16_pair(d[6][s], d[7][s]);
    *reinterpret_cast<uint4*>(row + s * slice_bytes + ((u ^ sw) << 4)) = w;
    w.x ^= 0x80008000u; w.y ^= 0x80008000u; w.z ^= 0x80008000u; w.w ^= 0x80008000u;
    *reinterpret_cast<uint4*>(nrow + s * slice_bytes + ((nu ^ sw) << 4)) = w;
  }
}

// ncp: columns per tile (multiple of 16, at most 64); nrt, nct row and column tiles; rr, rc their
// rows and columns.  upper: tiles strictly below the diagonal are left out.
template <int KA, int KB>
__global__ void __launch_bounds__(THREADS, 1)
    zgemm_tc64_kernel(ZOp A, ZOp B, double2* __restrict__ C, int* __restrict__ ec, int W, int n,
                      int ncp, int nrt, int nct, int rr, int rc, int upper, int accum,
                      DevStatus* st) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[2], empty[2], acc_full, acc_empty, done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b_slice = ncp * ROW_BYTES;
  unsigned char* sA = base;
  unsigned char* sB = base + ND * A_SLICE;
  const int nch = (W + CH - 1) / CH;
  const int per_k = nrt * nct;
  const int64_t n_tiles = (int64_t)n * per_k;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&full[s], STAGE_THREADS); mbar_init(&empty[s], 1); }
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, EPI_THREADS);
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base_sh)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  auto skip = [&](int in) { return upper && (in / nct) * rr >= (in % nct) * rc + rc; };

  if (warp < 8) {
    // ---------------- staging: threads 0-127 a row of A and half a chunk, 128-255 a column of B
    const int t = threadIdx.x;
    const bool is_b = t >= 128;
    const int r = is_b ? (t - 128) % ncp : t & 63;
    const int qg = is_b ? (t - 128) / ncp : t >> 6;
    const bool active = qg < 2;
    const int sw = r & 7;
    unsigned char* rowp = is_b ? sB + r * ROW_BYTES : sA + r * ROW_BYTES;
    int g = 0;
    bool ok = true;
    for (int64_t id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const int64_t k = id / per_k;
      const int in = (int)(id - k * per_k);
      if (skip(in)) continue;
      const int r0 = (in / nct) * rr, c0 = (in % nct) * rc;
      const int gr = is_b ? (r < rc ? c0 + r : W) : (r < rr ? r0 + r : W);
      const int e = is_b ? op_exp(B, k) : op_exp(A, k);
      for (int c = 0; c < nch; ++c, ++g) {
        const int h = g & 1;
        double2 v[8];
        if (active) {
          if (is_b) load8<KB>(B, k, W, true, gr, c * CH + 8 * qg, v);
          else load8<KA>(A, k, W, false, gr, c * CH + 8 * qg, v);
        }
        if (g >= 2 && !mbar_wait(&empty[h], ((uint32_t)(g >> 1) & 1u) ^ 1u)) ok = false;
        if (!ok || abort_sh) { ok = false; break; }
        if (active) {
          uint32_t d[8][ND];
          const int u = 4 * h + qg;
#pragma unroll
          for (int i = 0; i < 8; ++i) digits7(fixed55(v[i].x, e), d[i]);
          if (is_b) {
            put8(d, rowp, sw, b_slice, u);
          } else {
            put8(d, rowp, sw, A_SLICE, u);                            // Ar in the real row
            put8(d, rowp + 64 * ROW_BYTES, sw, A_SLICE, u + 2);       // Ar in the imaginary row
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) digits7(fixed55(v[i].y, e), d[i]);
          if (is_b) put8(d, rowp, sw, b_slice, u + 2);
          else put8_pm(d, rowp + 64 * ROW_BYTES, u, rowp, u + 2, sw, A_SLICE);   // Ai, and -Ai
        }
        fence_proxy_async_smem();
        mbar_arrive(&full[h]);
      }
    }
    if (!ok) {
      atomicOr(&st->bits, ST_TIMEOUT);
      abort_sh = 1;
    }
  } else {
    // ---------------- epilogue: warp w reads TMEM lanes 32 (w % 4) ..; half of the columns.  Warp 8
    // also issues the MMAs of a drain group, which cannot overlap a drain (the levels fill TMEM):
    // A_i against the stacked B_j, j <= min(6, 7 - i); columns of level i + j at (i + j) ncp
    int g = 0;
    const int per = 256 / ncp;   // slices per instruction (N <= 256)
    auto issue = [&](int c0, int c1, int G) -> bool {
      if (abort_sh || (G >= 1 && !mbar_wait(&acc_empty, (uint32_t)(G - 1) & 1u))) return false;
      for (int c = c0; c < c1; ++c, ++g) {
        const int h = g & 1;
        if (abort_sh || !mbar_wait(&full[h], (uint32_t)(g >> 1) & 1u)) return false;
        tc_fence_after();
#pragma unroll 1
        for (int kk = 0; kk < 2; ++kk) {
          const uint32_t off = (uint32_t)(64 * h + 32 * kk);
          const bool init = c == c0 && kk == 0;
#pragma unroll 1
          for (int i = 0; i < ND; ++i) {
            const uint64_t da = umma_desc_sw128(smem_u32(sA + i * A_SLICE) + off);
            const int nj = i == 0 ? ND : NLEV - i;   // slices j of B
            for (int j = 0; j < nj;) {
              // A_0 initialises the levels 0-6, A_1 B_6 level 7
              const bool seven = init && i == 1 && j == ND - 1;
              int m = min(per, nj - j);
              if (init && i == 1 && j < ND - 1) m = min(m, ND - 1 - j);
              const uint64_t db = umma_desc_sw128(smem_u32(sB + j * b_slice) + off);
              umma_bf16(tmem + (uint32_t)((i + j) * ncp), da, db, idesc_n(m * ncp),
                        (init && i == 0) || seven ? 0u : 1u);
              j += m;
            }
          }
        }
        umma_commit(&empty[h]);
      }
      umma_commit(&acc_full);
      return true;
    };
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane, cr = row & 63;
    const int part = row >> 6;   // 0: real part, 1: imaginary part
    const int half = (warp - 8) >> 2;
    const int c_lo = half * (ncp / 2);
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    bool ok = true;
    int G = 0;
    for (int64_t id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const int64_t k = id / per_k;
      const int in = (int)(id - k * per_k);
      if (skip(in)) continue;
      const int r0 = (in / nct) * rr, c0 = (in % nct) * rc;
      const int ea = op_exp(A, k), eb = op_exp(B, k);
      const bool bad = ea >= ZEXP_BAD || eb >= ZEXP_BAD;
      const int es = bad ? 0 : ea + eb - 55;
      const bool live = cr < rr && r0 + cr < W;
      double* Cr = reinterpret_cast<double*>(C + k * (int64_t)W * W + (int64_t)(live ? r0 + cr : 0) * W) + part;
      const int ncol = min(rc, W - c0);
      unsigned mx = 0u;
      for (int gi = 0; gi * GROUP < nch; ++gi, ++G) {
        if (warp == 8) {
          if (lane == 0) ok = issue(gi * GROUP, min(nch, (gi + 1) * GROUP), G);
          __syncwarp();
        }
        ok = ok && mbar_wait(&acc_full, (uint32_t)G & 1u);
        ok = __all_sync(0xffffffffu, ok && !abort_sh);   // tcgen05.ld is warp-collective
        if (!ok) break;
        tc_fence_after();
        const bool add = accum || gi > 0, final_group = (gi + 1) * GROUP >= nch;
#pragma unroll 1
        for (int cc = c_lo; cc < c_lo + ncp / 2; cc += 8) {
          uint32_t x[NLEV][8];
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_ld8_async(lane_addr + (uint32_t)(l * ncp + cc), x[l]);
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_wait_ld8(x[l]);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            int I[NLEV];
#pragma unroll
            for (int l = 0; l < NLEV; ++l) I[l] = __float2int_rn(__uint_as_float(x[l][j]));
            // sum_l I_l 2^(41 - 8 l), the levels 6 and 7 rounded to the unit 2^-55
            const long long hi = (long long)I[0] * 65536 + ((long long)I[1] * 256 + I[2]);
            const long long lo = (long long)I[3] * 65536 + ((long long)I[4] * 256 + I[5]);
            const long long t = (hi << 25) + (lo << 1) + (((long long)I[6] * 256 + (I[7] + 16384)) >> 15);
            const int col = cc + j;
            if (live && col < ncol) {
              double v = bad ? __longlong_as_double(0x7FF8000000000000ll) : int_to_double(t, es);
              double* dst = Cr + 2 * (int64_t)(c0 + col);
              if (add) v += *dst;
              *dst = v;
              if (final_group) mx = max(mx, (unsigned)(mag_bits(v) >> 32));
            }
          }
        }
        tc_fence_before();
        mbar_arrive(&acc_empty);
      }
      if (ec && ok) {
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int ex = (int)(mx >> 20);
        if (lane == 0) atomicMax(&ec[k], ex == 0x7FF ? ZEXP_BAD : ex - 1022);
      }
    }
    if (!ok) {
      atomicOr(&st->bits, ST_TIMEOUT);
      abort_sh = 1;
    }
    if (warp == 8 && lane == 0) umma_commit(&done_bar);   // all issued MMAs complete
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    if (lane == 0) mbar_wait(&done_bar, 0);
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

// e[k]: exponent above the largest of len doubles at x + k ld (ZEXP_BAD: infinite or NaN)
__global__ void __launch_bounds__(128) maxexp_kernel(const double* __restrict__ x, int64_t ld,
                                                     int len, int* __restrict__ e) {
  __shared__ unsigned s[4];
  const double* p = x + (int64_t)blockIdx.x * ld;
  unsigned m = 0u;
  for (int i = threadIdx.x; i < len; i += 128) m = max(m, (unsigned)(mag_bits(p[i]) >> 32));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    m = max(max(s[0], s[1]), max(s[2], s[3]));
    const int ex = (int)(m >> 20);
    e[blockIdx.x] = ex == 0x7FF ? ZEXP_BAD : ex - 1022;
  }
}

// ------------------------------------------------------------------ curvature
// One CTA per k-point.  The pairs n < m of rows n and W - 2 - n make W together, so a warp walks two
// rows at a time with every lane busy (a pair costs about 17 FP64 instructions, and one issues
// for 16 clocks whatever its active lanes); T_nm goes to shared memory and band n then adds row n
// and subtracts column n in order: T_mn = -T_nm exactly, and the sum is deterministic.
__global__ void __launch_bounds__(256) curvature64_kernel(const double* __restrict__ E,
                                                          const double2* __restrict__ Vx,
                                                          const double2* __restrict__ Vy, int W,
                                                          const double* __restrict__ etas, int n_eta,
                                                          double* __restrict__ Om,
                                                          int64_t eta_stride) {
  extern __shared__ double sT[];   // [W][W | 1]
  __shared__ double sE[128];
  __shared__ double s_emax;
  const int LD = W | 1;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t k = blockIdx.x;
  for (int j = t; j < W; j += 256) sE[j] = E[k * W + j];
  __syncthreads();
  if (warp == 0) {
    unsigned long long m = 0ull;
    for (int j = lane; j < W; j += 32) {
      const unsigned long long u = mag_bits(sE[j]);
      if (u <= 0x7FF0000000000000ull && u > m) m = u;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
      m = v > m ? v : m;
    }
    if (lane == 0) s_emax = __longlong_as_double((long long)m);
  }
  __syncthreads();
  const double thr2 = (1e-12 * s_emax) * (1e-12 * s_emax);
  const double2* X = Vx + k * (int64_t)W * W;
  const double2* Y = Vy + k * (int64_t)W * W;
  for (int e = 0; e < n_eta; ++e) {
    const double eta = etas[e];
    for (int n0 = warp; 2 * n0 <= W - 2; n0 += 8) {
      const int n1 = W - 2 - n0;                       // the partner row (n0 itself in the middle)
      const int len = W - 1 - n0, tot = n1 == n0 ? len : W;
      for (int p = lane; p < tot; p += 32) {
        const int n = p < len ? n0 : n1, m = p < len ? n0 + 1 + p : n1 + 1 + (p - len);
        const double2 x = X[n * W + m], y = Y[n * W + m];
        const double num = -2.0 * (x.y * y.x - x.x * y.y);
        const double dE = sE[n] - sE[m];
        const double d2 = dE * dE;
        sT[n * LD + m] = eta == 0.0 && d2 <= thr2 ? 0.0 : num / fma(eta, eta, d2);
      }
    }
    __syncthreads();
    // four lanes per band, each a strided part of the others, added in a fixed order
    for (int a0 = 0; a0 < W; a0 += 64) {
      const int a = a0 + (t >> 2);
      double s = 0.0;
      if (a < W)
        for (int m = t & 3; m < W; m += 4) {
          if (m > a) s += sT[a * LD + m];
          else if (m < a) s -= sT[m * LD + a];
        }
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (a < W && (t & 3) == 0) Om[e * eta_stride + k * W + a] = s;
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_maxexp(const double* x, int64_t ld, int len, int n, int* e, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  maxexp_kernel<<<n, 128, 0, s>>>(x, ld, len, e);
  return cudaGetLastError();
}

cudaError_t launch_zgemm_tc64(const ZOp& A, const ZOp& B, double2* C, int* ec, int W, int n, bool upper,
                              bool accum, DevStatus* st, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (W < 1 || W > LARGE_W_MAX || B.kind == 2) return cudaErrorInvalidValue;
  // even split of W into tiles of at most 64
  const int nt = (W + 63) / 64, rr = (W + nt - 1) / nt;
  const int ncp = (rr + 15) / 16 * 16;
  const size_t sm = (size_t)ND * A_SLICE + (size_t)ND * ncp * ROW_BYTES + 1024;
  int dev = 0, nsm = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    if (ec) {
      e = cudaMemsetAsync(ec, 0xC0, sizeof(int) * (size_t)n, s);   // a large negative exponent
      if (e != cudaSuccess) return e;
    }
    const int64_t tiles = (int64_t)n * nt * nt;
    kern<<<(int)std::min<int64_t>(tiles, std::max(nsm, 1)), THREADS, sm, s>>>(
        A, B, C, ec, W, n, ncp, nt, nt, rr, rr, upper ? 1 : 0, accum ? 1 : 0, st);
    return cudaGetLastError();
  };
  if (A.kind == 0) return B.kind == 0 ? go(zgemm_tc64_kernel<0, 0>) : go(zgemm_tc64_kernel<0, 1>);
  if (A.kind == 1) return B.kind == 0 ? go(zgemm_tc64_kernel<1, 0>) : cudaErrorInvalidValue;
  return B.kind == 0 ? go(zgemm_tc64_kernel<2, 0>) : cudaErrorInvalidValue;
}

cudaError_t launch_curvature64(const double* E, const double2* Vx, const double2* Vy, int W, int n,
                               const double* etas, int n_eta, double* Om, int64_t eta_stride,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (W > LARGE_W_MAX) return cudaErrorInvalidValue;
  const size_t sm = (size_t)W * (W | 1) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(curvature64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  curvature64_kernel<<<n, 256, sm, s>>>(E, Vx, Vy, W, etas, n_eta, Om, eta_stride);
  return cudaGetLastError();
}

}  // namespace kubo
