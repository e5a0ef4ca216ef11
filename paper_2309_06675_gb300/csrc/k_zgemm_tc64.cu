// Batched complex W x W products of FP64 grade on the 5th-generation tensor cores, W <= 128, and
// the curvature of Eq. 3 from the velocity matrices they form.
//
//   C[k] = op(A[k]) op(B[k]) (+ C[k]),  op: identity, conjugate transpose, or (A) a Hermitian matrix
//   from its packed real row
//
// Every real and imaginary part is cut into seven signed base-256 digits (FP16) relative to its matrix's
// largest entry (digits.cuh) and the digit products of the levels i + j <= 7 are kept (34 of 49, level
// 7 without the single pair that needs an eighth digit): the operands' rounding, 2^-56 of the largest
// entries, is the error that remains (levels 8 and beyond are 2^-65 per product).  A level sum over 128 of
// K is an integer of at most 7 x 128 x 2^14 < 2^24, exact in the FP32 accumulator.
//
// One tile is 64 complex rows by up to 64 columns as a real product [re; im] (M = 128) with K = 2 W:
// the rows [Ar | -Ai] and [Ai | Ar] against [Br; Bi].  A chunk is 16 of the inner index (32 of K); the
// staging warps load it in FP64, cut it and write it to shared memory (128-byte swizzle, a row of 64
// FP16 holding two chunks) while the MMAs of the other half run; the eight level sums of a
// tile fill the 512 TMEM columns (N = 64); eight warps add them in one int64 (units
// 2^-55 of the operand scales), convert, and write 16 columns at a time through shared memory.
//
// What bounds it: the MMAs (34 x 128 x N x 2 W / 4096 clocks per tile) and the staging of the next chunk
// (about 500 instructions for each 8 complex entries) take about the same time.  FP64 FMA kernels
// of the same products ran at 1.1 TFLOP/s; measured here: see the table beside the launcher.
//
// Every mbarrier wait is bounded; a wait that gives up sets ST_TIMEOUT and the CTA returns.
#include <algorithm>

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
constexpr int SLAB = 16;            // output columns written together
constexpr int E_MIN = -1080;        // exponent of an all-zero operand

__host__ __device__ __forceinline__ uint32_t idesc_n(int n) {
  // kind::f16, A = B = FP16, D = FP32, both K-major
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ int op_exp(const ZOp& o, int64_t k) { return o.e ? max(o.e[k], E_MIN) : 0; }

// v 2^e in FP64: the conversion is one instruction of the (here idle) FP64 pipe, the power of two an
// addition to the exponent field
__device__ __forceinline__ double scaled_double(long long v, int e) {
  const double d = (double)v;
  if (e < -900 || e > 900) return fx::scale_pow2(d, e);
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// ------------------------------------------------------------------ operand fetch
// A group of threads (128 for A, 2 ncp for B) brings one chunk of its operand, nrow rows (A) or columns
// (B) from g0 on by 16 inner indices from q0 on, into shared memory: entry (r, q) to slot
// raw[(q % 8) RAW_PITCH + r + nrow (q / 8)], where the thread that cuts row r's half chunk q / 8
// reads its eight entries without bank conflicts.  Asynchronous copies (zeros outside the matrix), the
// lanes along whichever index is contiguous in memory.
constexpr int RAW_PITCH = STAGE_THREADS + 1;
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES),
               "r"(on ? BYTES : 0)
               : "memory");
}
// lanes along the inner index: rows (t / 16) + RS i, index t % 16; mask: rows inside the matrix
template <int BYTES, int RS>
__device__ __forceinline__ void fetch_rows(const char* src, int64_t step, const char* safe, double2* dst,
                                           unsigned mask, bool on) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool g = on && ((mask >> i) & 1u);
    cp_async<BYTES>(dst + i * RS, g ? src : safe, g);
    src += step;
  }
}
// lanes along the rows: row t % nrow, inner indices (t / nrow) + 2 i, nq of them inside the matrix
template <int BYTES, int NROW>
__device__ __forceinline__ void fetch_cols(const char* src, int64_t step, const char* safe, char* dst, int nq) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool g = 2 * i < nq;
    cp_async<BYTES>(dst + (2 * (i & 3) * RAW_PITCH + NROW * (i >> 2)) * (int)sizeof(double2), g ? src : safe, g);
    src += step;
  }
}
// chunk c of rows (columns) g0 .. glim - 1 of an operand, NROW of them per tile, by 2 NROW threads
template <int NROW>
__device__ __forceinline__ void fetch_chunk(const ZOp& o, int64_t k, int W, bool is_b, int t, int g0, int glim,
                                            int c, double2* raw) {
  constexpr int RS = NROW / 8;
  const int rr = t >> 4, rq = t & 15;              // row-wise: first row, inner index
  const int cr = t % NROW, cq = t / NROW;          // column-wise: row, first inner index
  double2* rdst = raw + (rq & 7) * RAW_PITCH + rr + NROW * (rq >> 3);
  char* cdst = reinterpret_cast<char*>(raw + cq * RAW_PITCH + cr);
  const int left = glim - g0 - rr;                 // rows from rr on that exist
  const unsigned mask = left <= 0 ? 0u : left > 7 * RS ? 0xFFu : (1u << ((left + RS - 1) / RS)) - 1u;
  const bool ron = c * CH + rq < W;
  const int nq = g0 + cr < glim ? W - c * CH - cq : 0;
  if (o.kind == 2) {   // packed Hermitian rows: (P(r, q), P(q, r))
    const double* P = reinterpret_cast<const double*>(o.p) + k * o.ld;
    const char* safe = reinterpret_cast<const char*>(P);
    fetch_rows<8, RS>(reinterpret_cast<const char*>(P + (int64_t)(g0 + rr) * W + c * CH + rq), (int64_t)RS * W * 8,
                      safe, rdst, mask, ron);
    fetch_cols<8, NROW>(reinterpret_cast<const char*>(P + (int64_t)(c * CH + cq) * W + g0 + cr), (int64_t)2 * W * 8,
                        safe, cdst + 8, nq);
    return;
  }
  // A: (r, q) of the matrix or, conjugated, (q, r); B: (q, r) or, conjugated, (r, q)
  const double2* P = reinterpret_cast<const double2*>(o.p) + k * (int64_t)W * W;
  const char* safe = reinterpret_cast<const char*>(P);
  if ((o.kind == 0) != is_b)
    fetch_rows<16, RS>(reinterpret_cast<const char*>(P + (int64_t)(g0 + rr) * W + c * CH + rq),
                       (int64_t)RS * W * 16, safe, rdst, mask, ron);
  else
    fetch_cols<16, NROW>(reinterpret_cast<const char*>(P + (int64_t)(c * CH + cq) * W + g0 + cr),
                         (int64_t)2 * W * 16, safe, cdst, nq);
}
// round(x 2^(55 - e)) for |x| <= 2^e with e2 = e + 1030 and e above -900 (zeros and subnormals are then
// far below the unit): the general form without its case distinctions
__device__ __forceinline__ long long fixed55_mid(double x, int e2) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int s = min(e2 - (int)((hi >> 20) & 0x7FFu) - 1, 63);
  const unsigned long long m = ((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32 | lo) << 10;
  const long long q = (long long)(((m >> s) + 1ull) >> 1);
  const long long sg = (long long)((int)hi >> 31);
  return (q ^ sg) - sg;
}
// a thread's eight fetched entries (row gr, inner indices q0 ..) as fixed-point parts (55 fractional
// bits below 2^e)
__device__ __forceinline__ void take8(const double2* slot, int kind, int gr, int q0, int e,
                                      long long (&re)[8], long long (&im)[8]) {
  const bool mid = e > -900;   // (the same for all threads of an operand)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    double2 v = slot[i * RAW_PITCH];
    // Hermitian: (a, b) = packed (r, q) and (q, r); Re is the one above the diagonal
    if (kind == 2) v = gr < q0 + i ? v : gr > q0 + i ? make_double2(v.y, -v.x) : make_double2(v.x, 0.0);
    if (kind == 1) v.y = __hiloint2double(__double2hiint(v.y) ^ (int)0x80000000, __double2loint(v.y));
    re[i] = mid ? fixed55_mid(v.x, e + 1030) : fixed55(v.x, e);
    im[i] = mid ? fixed55_mid(v.y, e + 1030) : fixed55(v.y, e);
  }
}

// the seven digit slices of 8 values at 16-byte unit u of a row; TWO: also at unit u2 of a second row,
// NEG with the opposite sign
template <bool TWO, bool NEG>
__device__ __forceinline__ void put8(const long long (&q)[8], unsigned char* row, int u, unsigned char* row2,
                                     int u2, int sw, int slice_bytes) {
  uint32_t d[4][ND];
#pragma unroll
  for (int i = 0; i < 4; ++i) digits7_h2(q[2 * i], q[2 * i + 1], d[i]);
#pragma unroll
  for (int s = 0; s < ND; ++s) {
    *reinterpret_cast<uint4*>(row + s * slice_bytes + ((u ^ sw) << 4)) = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
    if (TWO)
      *reinterpret_cast<uint4*>(row2 + s * slice_bytes + ((u2 ^ sw) << 4)) =
          NEG ? make_uint4(h2_sub(0u, d[0][s]), h2_sub(0u, d[1][s]), h2_sub(0u, d[2][s]), h2_sub(0u, d[3][s]))
              : make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
  }
}

// One K16 step: A_i against the stacked B_j, j <= min(6, 7 - i), into the columns of the levels i + j (at
// (i + j) NCP).  Straight-line code with constant offsets: with the descriptors computed in a loop
// the issuing lane took about 200 clocks per MMA, twice what the MMAs themselves take.
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);   // as umma_desc_sw128
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tmov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(d),
      "r"(alo), "r"(blo), "r"(idesc), "r"((uint32_t)acc), "r"(DESC_HI)
      : "memory");
}
template <int NCP, bool INIT>
__device__ __forceinline__ void mma_step(uint32_t tmem, uint32_t alo, uint32_t blo) {
  constexpr int PER = 256 / NCP;   // slices per instruction (N <= 256)
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    // INIT: A_0 initialises the levels 0-6 and A_1 B_6 level 7
    const int nj = i == 0 ? ND : NLEV - i;
    const int cut = INIT && i == 1 ? ND - 1 : nj;
#pragma unroll
    for (int j = 0; j < ND; j += PER)
      if (j < cut) {
        const int m = cut - j < PER ? cut - j : PER;
        mma_f16(tmem + (uint32_t)((i + j) * NCP), alo + i * (A_SLICE >> 4), blo + j * (NCP * ROW_BYTES >> 4),
                idesc_n(m * NCP), !(INIT && i == 0));
      }
    if (INIT && i == 1)
      mma_f16(tmem + (uint32_t)(ND * NCP), alo + i * (A_SLICE >> 4), blo + (ND - 1) * (NCP * ROW_BYTES >> 4),
              idesc_n(NCP), false);
  }
}

// NCP: columns per tile; nrt, nct row and column tiles of rr rows and columns.  upper: tiles strictly
// below the diagonal are left out.
template <int NCP>
__global__ void __launch_bounds__(THREADS, 1)
    zgemm_tc64_kernel(ZOp A, ZOp B, double2* __restrict__ C, int* __restrict__ ec, int W, int n,
                      int nrt, int rr, int upper, int accum, DevStatus* st) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[2], empty[2], acc_full, acc_empty, done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_sh, leave_sh, leave_epi_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int B_SLICE = NCP * ROW_BYTES;
  unsigned char* sA = base;
  unsigned char* sB = sA + ND * A_SLICE;
  double2* raw0 = reinterpret_cast<double2*>(sB + ND * B_SLICE);
  double2* slab = raw0 + 8 * RAW_PITCH;   // [64 rows][SLAB + 1]: a slab of output columns
  const int nch = (W + CH - 1) / CH;
  const int per_k = nrt * nrt;
  const int64_t n_tiles = (int64_t)n * per_k;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&full[s], STAGE_THREADS); mbar_init(&empty[s], 1); }
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, EPI_THREADS);
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    leave_sh = 0;
    leave_epi_sh = 0;
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
  auto skip = [&](int in) { return upper && in / nrt > in % nrt; };

  if (warp < 8) {
    // ---------------- staging: threads 0-127 a row of A and half a chunk, 128-255 a column of B
    const bool is_b = threadIdx.x >= 128;
    const int t = threadIdx.x & 127;
    const int nrow = is_b ? NCP : 64, nthr = is_b ? 2 * NCP : 128;
    const int r = is_b ? t % NCP : t & 63, qg = is_b ? t / NCP : t >> 6;
    const bool active = t < nthr;
    const int sw = r & 7;
    unsigned char* rowp = (is_b ? sB : sA) + r * ROW_BYTES;
    double2* raw = raw0 + (is_b ? 128 : 0);
    const ZOp& O = is_b ? B : A;
    int g = 0;
    bool ok = true;
    // the chunk being fetched: tile id, its matrix, the operand's first row there, exponent
    int64_t id = blockIdx.x, k = 0;
    int g0 = 0, e = 0, c = 0;
    auto enter = [&]() {   // the next tile to be worked on, from id on
      while (id < n_tiles && skip((int)(id % per_k))) id += gridDim.x;
      if (id >= n_tiles) return;
      k = id / per_k;
      const int in = (int)(id - k * per_k);
      g0 = (is_b ? in % nrt : in / nrt) * rr;
      e = op_exp(O, k);
    };
    auto fetch = [&]() {
      if (id < n_tiles && active) {
        if (is_b) fetch_chunk<NCP>(O, k, W, true, t, g0, min(W, g0 + rr), c, raw);
        else fetch_chunk<64>(O, k, W, false, t, g0, min(W, g0 + rr), c, raw);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    enter();
    fetch();
    while (id < n_tiles) {
      const int h = g & 1;
      long long re[8], im[8];
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      asm volatile("bar.sync 1, 256;" ::: "memory");   // the chunk is complete
      const bool stop = abort_sh != 0;
      if (active) take8(raw + r + nrow * qg, O.kind, g0 + r, c * CH + 8 * qg, e, re, im);
      if (stop) leave_sh = 1;
      asm volatile("bar.sync 1, 256;" ::: "memory");   // its slots may be overwritten
      if (leave_sh) break;                             // (all of them, after a timeout anywhere)
      if (++c == nch) {
        c = 0;
        id += gridDim.x;
        enter();
      }
      fetch();
      if (g >= 2 && !mbar_wait(&empty[h], ((uint32_t)(g >> 1) & 1u) ^ 1u)) {
        atomicOr(&st->bits, ST_TIMEOUT);   // (go on: every warp passes the same barriers)
        abort_sh = 1;
        ok = false;
      }
      if (active && ok) {
        const int u = 4 * h + qg;
        if (is_b) {
          put8<false, false>(re, rowp, u, rowp, u, sw, B_SLICE);
          put8<false, false>(im, rowp, u + 2, rowp, u, sw, B_SLICE);
        } else {   // real rows [Ar | -Ai], imaginary rows [Ai | Ar]
          unsigned char* rowi = rowp + 64 * ROW_BYTES;
          put8<true, false>(re, rowp, u, rowi, u + 2, sw, A_SLICE);
          put8<true, true>(im, rowi, u, rowp, u + 2, sw, A_SLICE);
        }
      }
      fence_proxy_async_smem();
      mbar_arrive(&full[h]);
      ++g;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else {
    // ---------------- epilogue: warp w reads TMEM lanes 32 (w % 4) .. and, per slab of 16 columns, 8 of
    // them.  Warp 8 also issues the MMAs of a drain group, which cannot overlap a drain (the levels
    // fill TMEM).
    int g = 0;
    auto issue = [&](int nc, int G) -> bool {
      if (abort_sh || (G >= 1 && !mbar_wait(&acc_empty, (uint32_t)(G - 1) & 1u))) return false;
      const uint32_t a0 = ((smem_u32(sA) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t b0 = ((smem_u32(sB) & 0x3FFFFu) >> 4) | (1u << 16);
#pragma unroll 1
      for (int c = 0; c < nc; ++c, ++g) {
        const uint32_t off = (uint32_t)(g & 1) * 4u;   // (64 bytes: the chunk's half of a row)
        if (abort_sh || !mbar_wait(&full[g & 1], (uint32_t)(g >> 1) & 1u)) return false;
        tc_fence_after();
        if (c == 0) mma_step<NCP, true>(tmem, a0 + off, b0 + off);
        else mma_step<NCP, false>(tmem, a0 + off, b0 + off);
        mma_step<NCP, false>(tmem, a0 + off + 2, b0 + off + 2);
        umma_commit(&empty[g & 1]);
      }
      umma_commit(&acc_full);
      return true;
    };
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane, cr = row & 63;
    const int part = row >> 6;   // 0: real part, 1: imaginary part
    const int half = (warp - 8) >> 2;
    const int et = threadIdx.x - STAGE_THREADS;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    bool ok = true;
    int G = 0;
    for (int64_t id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      const int64_t k = id / per_k;
      const int in = (int)(id - k * per_k);
      if (skip(in)) continue;
      const int r0 = (in / nrt) * rr, c0 = (in % nrt) * rr;
      const int ea = op_exp(A, k), eb = op_exp(B, k);
      const bool bad = ea >= ZEXP_BAD || eb >= ZEXP_BAD;
      const int es = bad ? 0 : ea + eb - 55;
      const int nrow = min(rr, W - r0), ncol = min(rr, W - c0);
      double2* Ck = C + k * (int64_t)W * W + (int64_t)r0 * W + c0;
      unsigned mx = 0u;
      for (int gi = 0; gi * GROUP < nch; ++gi, ++G) {
        if (warp == 8) {
          if (lane == 0) ok = issue(min(GROUP, nch - gi * GROUP), G);
          __syncwarp();
        }
        ok = ok && mbar_wait(&acc_full, (uint32_t)G & 1u);
        ok = __all_sync(0xffffffffu, ok && !abort_sh);   // tcgen05.ld is warp-collective
        if (!ok) leave_epi_sh = 1;
        asm volatile("bar.sync 2, 256;" ::: "memory");
        if (leave_epi_sh) ok = false;
        asm volatile("bar.sync 2, 256;" ::: "memory");   // (every epilogue warp leaves together)
        if (!ok) break;
        tc_fence_after();
        const bool add = accum || gi > 0, final_group = (gi + 1) * GROUP >= nch;
#pragma unroll 1
        for (int s0 = 0; s0 < NCP; s0 += SLAB) {
          uint32_t x[NLEV][8];
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_ld8_async(lane_addr + (uint32_t)(l * NCP + s0 + 8 * half), x[l]);
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_wait_ld8(x[l]);
          if (s0 + SLAB >= NCP) {   // the thread's last TMEM read of this drain
            tc_fence_before();
            mbar_arrive(&acc_empty);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            int I[NLEV];
#pragma unroll
            for (int l = 0; l < NLEV; ++l) I[l] = __float2int_rn(__uint_as_float(x[l][j]));
            // sum_l I_l 2^(41 - 8 l), the levels 6 and 7 rounded to the unit 2^-55
            const long long hi = (long long)I[0] * 65536 + ((long long)I[1] * 256 + I[2]);
            const long long lo = (long long)I[3] * 65536 + ((long long)I[4] * 256 + I[5]);
            const long long v = (hi << 25) + (lo << 1) + (((long long)I[6] * 256 + (I[7] + 16384)) >> 15);
            reinterpret_cast<double*>(slab + cr * (SLAB + 1) + 8 * half + j)[part] =
                bad ? __longlong_as_double(0x7FF8000000000000ll) : scaled_double(v, es);
          }
          asm volatile("bar.sync 2, 256;" ::: "memory");
          // the slab to global memory, 16 columns (256 bytes) of a row by 16 lanes
#pragma unroll
          for (int q = 0; q < 64 * SLAB / EPI_THREADS; ++q) {
            const int rw = (et >> 4) + q * (EPI_THREADS / SLAB), cl = et & 15;
            if (rw < nrow && s0 + cl < ncol) {
              double2 v = slab[rw * (SLAB + 1) + cl];
              double2* dst = Ck + (int64_t)rw * W + s0 + cl;
              if (add) {
                const double2 o = *dst;
                v.x += o.x;
                v.y += o.y;
              }
              *dst = v;
              if (final_group) mx = max(mx, (unsigned)(max(mag_bits(v.x), mag_bits(v.y)) >> 32));
            }
          }
          asm volatile("bar.sync 2, 256;" ::: "memory");
        }
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
  const size_t sm = (size_t)ND * A_SLICE + (size_t)ND * ncp * ROW_BYTES +
                    ((size_t)8 * RAW_PITCH + 64 * (SLAB + 1)) * sizeof(double2) + 1024;
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
    kern<<<(int)std::min<int64_t>(tiles, std::max(nsm, 1)), THREADS, sm, s>>>(A, B, C, ec, W, n, nt, rr,
                                                                              upper ? 1 : 0, accum ? 1 : 0, st);
    return cudaGetLastError();
  };
  switch (ncp) {
    case 16: return go(zgemm_tc64_kernel<16>);
    case 32: return go(zgemm_tc64_kernel<32>);
    case 48: return go(zgemm_tc64_kernel<48>);
    default: return go(zgemm_tc64_kernel<64>);
  }
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
