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
// the rows [Ar | -Ai] and [Ai | Ar] against [Br; Bi].  A chunk is 8 of the inner index (K = 16); two groups
// of staging warps take the chunks in turn: load in FP64, cut, write to shared memory (128-byte swizzle, a
// row of 64 FP16 holding four chunks) while the MMAs of the chunks before run.  The eight level
// sums of a tile fill the 512 TMEM columns (N = 64); eight warps, each with both parts of 16
// complex rows in its lanes, add them in one int64 (units 2^-55 of the operand scales), convert, and write 8
// columns at a time through shared memory of their own.
//
// What bounds it: a tile of W = 64 takes 16.8 us, where its MMAs (34 x 128 x N x 2 W / 4096 clocks) take 4.6,
// the staging alone 12 (integer instructions at 44 % of their rate, the rest waits for loads and
// between its steps) and the drain alone 9; the drain cannot overlap the MMAs, which need all of TMEM.
// (One staging group with 16-index chunks and slabs shared by the eight drain warps: 20.8 us.)
// W = 64, 4,096 k-points: the four products and the curvature take 2.2 ms (FP64 FMA kernels of the same
// products ran at 1.1 TFLOP/s); W = 97, 2,744: 9.1 ms.
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
constexpr int CH = 8;               // inner indices per chunk (K = 16)
constexpr int NSLOT = 4;            // chunks in shared memory: 32 bytes each of a row
constexpr int GROUP = 8;            // chunks per drain (K = 128)
constexpr int NLEV = 8;
constexpr int ROW_BYTES = 128;      // 64 FP16: four chunks
constexpr int A_SLICE = BM * ROW_BYTES;          // 16 KB
constexpr int STAGE_THREADS = 512;  // two groups of 256, alternate chunks
constexpr int EPI_THREADS = 256;
constexpr int MMA_WARP = (STAGE_THREADS + EPI_THREADS) / 32;
constexpr int THREADS = STAGE_THREADS + EPI_THREADS + 32;   // 25 warps: 80 registers each
constexpr int TMEM_COLS = 512;
constexpr int SLAB = 8;             // output columns written together
constexpr int E_MIN = -1080;        // exponent of an all-zero operand

__host__ __device__ __forceinline__ uint32_t idesc_n(int n) {
  // kind::f16, A = B = FP16, D = FP32, both K-major
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ int op_exp(const ZOp& o, int64_t k) { return o.e ? max(o.e[k], E_MIN) : 0; }

// v 2^e in FP64: the conversion runs on the (here idle) FP64 pipe, the power of two is an addition to the
// exponent field (converting in integer instructions: 8 % more instructions, the same time)
__device__ __forceinline__ double scaled_double(long long v, int e) {
  const double d = (double)v;
  if (e < -900 || e > 900) return fx::scale_pow2(d, e);
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// ------------------------------------------------------------------ operand fetch
// Half a staging group (128 threads for A, 2 ncp for B) brings one chunk of its operand, nrow rows (A) or
// columns (B) from g0 on by 8 inner indices, into shared memory: entry (r, q) to slot
// raw[q RAW_PITCH + r], where the threads that cut row r read its eight entries without bank conflicts.
// Asynchronous copies (zeros outside the matrix), the lanes along whichever index is contiguous in
// memory.
constexpr int RAW_PITCH = 129;   // 64 rows of A and up to 64 columns of B
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES),
               "r"(on ? BYTES : 0)
               : "memory");
}
// lanes along the inner index: rows (t / 8) + RS i, index t % 8; mask: rows inside the matrix; the steps
// after an even and after an odd row
template <int BYTES, int RS>
__device__ __forceinline__ void fetch_rows(const char* src, int64_t step0, int64_t step1, const char* safe,
                                           double2* dst, unsigned mask, bool on) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool g = on && ((mask >> i) & 1u);
    cp_async<BYTES>(dst + i * RS, g ? src : safe, g);
    src += i & 1 ? step1 : step0;
  }
}
// lanes along the rows: row t % nrow, inner indices (t / nrow) + 2 i, nq of them inside the matrix
template <int BYTES>
__device__ __forceinline__ void fetch_cols(const char* src, int64_t step, const char* safe, char* dst, int nq) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool g = 2 * i < nq;
    cp_async<BYTES>(dst + 2 * i * RAW_PITCH * (int)sizeof(double2), g ? src : safe, g);
    src += step;
  }
}
// chunk c of rows (columns) g0 .. glim - 1 of an operand, NROW of them per tile, by 2 NROW threads.  Sources:
// A (r, q) of the matrix or, conjugated, (q, r); B (q, r) or, conjugated, (r, q); packed Hermitian rows (kind 2)
// P(r, q) and P(q, r)
template <int NROW>
__device__ __forceinline__ void fetch_chunk(const ZOp& o, int64_t k, int W, bool is_b, int t, int g0, int glim,
                                            int c, double2* raw) {
  constexpr int RS = NROW / 4;
  const int rr = t >> 3, rq = t & 7;               // row-wise: first row, inner index
  const int cr = t % NROW, cq = t / NROW;          // column-wise: row, first inner index
  double2* rdst = raw + rq * RAW_PITCH + rr;
  char* cdst = reinterpret_cast<char*>(raw + cq * RAW_PITCH + cr);
  const int left = glim - g0 - rr;                 // rows from rr on that exist
  const unsigned mask = left <= 0 ? 0u : left > 3 * RS ? 0xFu : (1u << ((left + RS - 1) / RS)) - 1u;
  const bool ron = c * CH + rq < W;
  const int nq = g0 + cr < glim ? W - c * CH - cq : 0;
  if (o.kind == 2) {
    const double* P = reinterpret_cast<const double*>(o.p) + k * o.ld;
    const char* safe = reinterpret_cast<const char*>(P);
    const int64_t step = (int64_t)RS * W * 8;
    fetch_rows<8, RS>(reinterpret_cast<const char*>(P + (int64_t)(g0 + rr) * W + c * CH + rq), step, step, safe,
                      rdst, mask, ron);
    fetch_cols<8>(reinterpret_cast<const char*>(P + (int64_t)(c * CH + cq) * W + g0 + cr), (int64_t)2 * W * 8,
                  safe, cdst + 8, nq);
    return;
  }
  const double2* P = reinterpret_cast<const double2*>(o.p) + k * (int64_t)W * W;
  const char* safe = reinterpret_cast<const char*>(P);
  const int64_t step = (int64_t)RS * W * 16;
  if ((o.kind == 0) != is_b)
    fetch_rows<16, RS>(reinterpret_cast<const char*>(P + (int64_t)(g0 + rr) * W + c * CH + rq), step, step, safe,
                       rdst, mask, ron);
  else
    fetch_cols<16>(reinterpret_cast<const char*>(P + (int64_t)(c * CH + cq) * W + g0 + cr), (int64_t)2 * W * 16,
                   safe, cdst, nq);
}
// the same for a tile of P matrices k .. k + P - 1 (below n), 64 / P of its rows (columns) each
template <int P>
__device__ __forceinline__ void fetch_chunk_packed(const ZOp& o, int64_t k, int n, int W, bool is_b, int t, int c,
                                                   double2* raw) {
  constexpr int RS = 16, SUB = 64 / P;
  const int rr = t >> 3, rq = t & 7, cr = t & 63, cq = t >> 6;
  const int csub = cr / SUB, cl = cr % SUB;
  const int left = (int)min((int64_t)P, n - k);    // matrices of the tile that exist
  unsigned mask = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) mask |= ((rr + RS * i) % SUB < W && (rr + RS * i) / SUB < left ? 1u : 0u) << i;
  const bool ron = c * CH + rq < W;
  const int nq = cl < W && csub < left ? W - c * CH - cq : 0;
  const int64_t bytes = o.kind == 2 ? 8 : 16, mat = o.kind == 2 ? o.ld * 8 : (int64_t)W * W * 16;
  const int64_t rows = (int64_t)RS * W * bytes;
  const int64_t s0 = P == 4 ? mat : rows, s1 = P == 4 ? mat : mat - rows;
  const char* base = reinterpret_cast<const char*>(o.p) + k * mat;
  const char* rsrc = base + ((int64_t)rr * W + c * CH + rq) * bytes;
  const char* csrc = base + csub * mat + ((int64_t)(c * CH + cq) * W + cl) * bytes;
  double2* rdst = raw + rq * RAW_PITCH + rr;
  char* cdst = reinterpret_cast<char*>(raw + cq * RAW_PITCH + cr);
  if (o.kind == 2) {
    fetch_rows<8, RS>(rsrc, s0, s1, base, rdst, mask, ron);
    fetch_cols<8>(csrc, (int64_t)2 * W * 8, base, cdst + 8, nq);
  } else if ((o.kind == 0) != is_b) {
    fetch_rows<16, RS>(rsrc, s0, s1, base, rdst, mask, ron);
  } else {
    fetch_cols<16>(csrc, (int64_t)2 * W * 16, base, cdst, nq);
  }
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
// the real (part 0) or imaginary parts of eight fetched entries (row gr, inner indices q0 ..) in fixed point
// (55 fractional bits below 2^e)
__device__ __forceinline__ void take8(const double* slot, int kind, int part, int gr, int q0, int e,
                                      long long (&v)[8]) {
  double x[8];
  if (kind == 2) {   // Hermitian, (a, b) = packed (r, q) and (q, r): Re is the one above the diagonal
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int d = gr - q0 - i;
      x[i] = slot[2 * i * RAW_PITCH + (d > 0 ? 1 - part : part)];
      if (part) x[i] = d == 0 ? 0.0 : d > 0 ? -x[i] : x[i];
    }
  } else {
    const int conj = kind == 1 && part ? (int)0x80000000 : 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      x[i] = slot[2 * i * RAW_PITCH + part];
      x[i] = __hiloint2double(__double2hiint(x[i]) ^ conj, __double2loint(x[i]));
    }
  }
  if (e > -900) {   // (the same for all threads of an operand)
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = fixed55_mid(x[i], e + 1030);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = fixed55(x[i], e);
  }
}

// the seven digit slices of 8 values at 16-byte unit u of a row; TWO: also at unit u2 of a second row,
// with the sign bits flipped by neg
template <bool TWO>
__device__ __forceinline__ void put8(const long long (&q)[8], unsigned char* row, int u, unsigned char* row2,
                                     int u2, uint32_t neg, int sw, int slice_bytes) {
  uint32_t d[4][ND];
#pragma unroll
  for (int i = 0; i < 4; ++i) digits7_h2(q[2 * i], q[2 * i + 1], d[i]);
#pragma unroll
  for (int s = 0; s < ND; ++s) {
    *reinterpret_cast<uint4*>(row + s * slice_bytes + ((u ^ sw) << 4)) = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
    if (TWO)
      *reinterpret_cast<uint4*>(row2 + s * slice_bytes + ((u2 ^ sw) << 4)) =
          make_uint4(d[0][s] ^ neg, d[1][s] ^ neg, d[2][s] ^ neg, d[3][s] ^ neg);
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
// below the diagonal are left out.  P > 1 (NCP = 64): P matrices of up to 64 / P rows share a tile, whose P
// diagonal blocks are drained.
template <int NCP, int P>
__global__ void __launch_bounds__(THREADS, 1)
    zgemm_tc64_kernel(ZOp A, ZOp B, double2* __restrict__ C, int* __restrict__ ec, int W, int n,
                      int nrt, int rr, int upper, int accum, DevStatus* st) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[NSLOT], empty[NSLOT], acc_full, acc_empty, done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_sh, leave_sh[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int B_SLICE = NCP * ROW_BYTES;
  unsigned char* sA = base;
  unsigned char* sB = sA + ND * A_SLICE;
  double2* raw0 = reinterpret_cast<double2*>(sB + ND * B_SLICE);
  double2* slab0 = raw0 + 2 * CH * RAW_PITCH;   // per epilogue warp [16 rows][SLAB + 1]: a slab of output columns
  const int nch = (W + CH - 1) / CH;
  // tile id: k-point, then row and column tile (nrt = 1 or 2 of them)
  const int lg = nrt - 1, n_tiles = P == 1 ? n << (2 * lg) : (n + P - 1) / P;
  constexpr int SUB = 64 / P, DRAIN_COLS = P == 1 ? NCP : SUB;
  auto row_of = [&](int id) { return (id >> lg) & lg; };
  auto col_of = [&](int id) { return id & lg; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSLOT; ++s) { mbar_init(&full[s], STAGE_THREADS / 2); mbar_init(&empty[s], 1); }
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, EPI_THREADS);
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    leave_sh[0] = leave_sh[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
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
  auto skip = [&](int id) { return upper && row_of(id) > col_of(id); };

  if (warp < STAGE_THREADS / 32) {
    // ---------------- staging: two groups of 256 threads, chunks g = group, group + 2, ... of the CTA's
    // sequence; in a group, threads 0-127 the real or imaginary parts of a row of A, 128-255 of a
    // column of B
    const int grp = threadIdx.x >> 8;
    const bool is_b = (threadIdx.x & 128) != 0;
    const int t = threadIdx.x & 127;
    const int nrow = is_b ? NCP : 64;
    const int r = is_b ? t % NCP : t & 63, part = is_b ? t / NCP : t >> 6;
    const bool active = t < 2 * nrow;
    const int sw = r & 7;
    // row of A: [re; im] in blocks of 16 (an epilogue warp's 32 lanes hold both parts of 16 rows)
    unsigned char* rowp = is_b ? sB + r * ROW_BYTES : sA + (32 * (r >> 4) + (r & 15)) * ROW_BYTES;
    double2* raw = raw0 + grp * CH * RAW_PITCH + (is_b ? 64 : 0);
    const ZOp& O = is_b ? B : A;
    auto sync = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + grp) : "memory"); };
    bool ok = true;
    // the chunk being fetched: tile id, its matrix, the operand's first row there, exponent
    const int sub = P == 1 ? 0 : r / SUB, rl = P == 1 ? r : r % SUB;   // matrix of the tile, row in it
    int id = blockIdx.x, k = 0;
    int g0 = 0, e = 0, c = 0;
    auto enter = [&]() {   // the next tile to be worked on, from id on
      while (id < n_tiles && skip(id)) id += gridDim.x;
      if (id >= n_tiles) return;
      k = (id >> (2 * lg)) * P;
      g0 = (is_b ? col_of(id) : row_of(id)) * rr;
      e = op_exp(O, P == 1 ? k : min(k + sub, n - 1));
    };
    auto advance = [&]() {
      if (id < n_tiles && ++c == nch) {
        c = 0;
        id += gridDim.x;
        enter();
      }
    };
    auto fetch = [&]() {
      if (id < n_tiles && active) {
        if constexpr (P > 1) fetch_chunk_packed<P>(O, k, n, W, is_b, t, c, raw);
        else if (is_b) fetch_chunk<NCP>(O, k, W, true, t, g0, min(W, g0 + rr), c, raw);
        else fetch_chunk<64>(O, k, W, false, t, g0, min(W, g0 + rr), c, raw);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    enter();
    if (grp) advance();
    fetch();
    for (int g = grp; id < n_tiles; g += 2) {
      const int h = g & (NSLOT - 1);
      long long v[8];
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      sync();   // the chunk is complete
      const bool stop = abort_sh != 0;
      if (active) take8(reinterpret_cast<const double*>(raw + r), O.kind, part, g0 + rl, c * CH, e, v);
      if (stop) leave_sh[grp] = 1;
      sync();                      // its slots may be overwritten
      if (leave_sh[grp]) break;    // (all of the group, after a timeout anywhere)
      advance();
      advance();
      fetch();
      if (g >= NSLOT && !mbar_wait(&empty[h], ((uint32_t)(g / NSLOT) & 1u) ^ 1u)) {
        atomicOr(&st->bits, ST_TIMEOUT);   // (go on: every warp passes the same barriers)
        abort_sh = 1;
        ok = false;
      }
      if (active && ok) {
        if (is_b) {
          put8<false>(v, rowp, 2 * h + part, rowp, 0, 0u, sw, B_SLICE);
        } else {   // real rows [Ar | -Ai], imaginary rows [Ai | Ar]
          unsigned char* rowi = rowp + 16 * ROW_BYTES;
          put8<true>(v, part ? rowi : rowp, 2 * h, part ? rowp : rowi, 2 * h + 1, part ? 0x80008000u : 0u, sw, A_SLICE);
        }
      }
      fence_proxy_async_smem();
      mbar_arrive(&full[h]);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  } else if (warp == MMA_WARP) {
    // ---------------- the MMAs, from one lane; a drain group waits for the drain before it (the levels
    // fill TMEM)
    if (lane == 0) {
      const uint32_t a0 = ((smem_u32(sA) & 0x3FFFFu) >> 4) | (1u << 16);
      const uint32_t b0 = ((smem_u32(sB) & 0x3FFFFu) >> 4) | (1u << 16);
      bool ok = true;
      int g = 0, G = 0;
      for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
        if (skip(id)) continue;
        for (int gi = 0; gi * GROUP < nch && ok; ++gi, ++G) {
          const int nc = min(GROUP, nch - gi * GROUP);
          ok = !abort_sh && (G == 0 || mbar_wait(&acc_empty, (uint32_t)(G - 1) & 1u));
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < nc && ok; ++c, ++g) {
            const int h = g & (NSLOT - 1);
            const uint32_t off = (uint32_t)h * 2u;   // (32 bytes: the chunk's quarter of a row)
            ok = !abort_sh && mbar_wait(&full[h], (uint32_t)(g / NSLOT) & 1u);
            if (!ok) break;
            tc_fence_after();
            if (c == 0) mma_step<NCP, true>(tmem, a0 + off, b0 + off);
            else mma_step<NCP, false>(tmem, a0 + off, b0 + off);
            umma_commit(&empty[h]);
          }
          if (ok) umma_commit(&acc_full);
        }
      }
      if (!ok) {
        atomicOr(&st->bits, ST_TIMEOUT);
        abort_sh = 1;
      }
      umma_commit(&done_bar);   // all issued MMAs complete
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: warp w reads the TMEM lanes 32 (w % 4) .., both parts of 16 complex rows,
    // and every other slab of 8 columns, and writes it through shared memory of its own
    const int quarter = warp & 3, half = (warp - STAGE_THREADS / 32) >> 2;
    const int wr = lane >> 3, wc = lane & 7;   // writes rows wr + 4 q of a slab's column wc
    double2* slab = slab0 + (warp - STAGE_THREADS / 32) * 16 * (SLAB + 1);
    double* mine = reinterpret_cast<double*>(slab + (lane & 15) * (SLAB + 1)) + (lane >> 4);
    const int sub = P == 1 ? 0 : 16 * quarter / SUB;                  // matrix of the tile
    const int ro = P == 1 ? 16 * quarter : (16 * quarter) % SUB;      // row in it
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(sub * SUB);
    bool ok = true;
    int G = 0;
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      if (skip(id)) continue;
      const int k1 = (id >> (2 * lg)) * P + sub;
      const int64_t k = P == 1 ? k1 : min(k1, n - 1);
      const int r0 = row_of(id) * rr + ro, c0 = col_of(id) * rr;
      const int ea = op_exp(A, k), eb = op_exp(B, k);
      const bool bad = ea >= ZEXP_BAD || eb >= ZEXP_BAD;
      const int es = bad ? 0 : ea + eb - 55;
      const int nrow = P == 1 || k1 < n ? min(rr - ro, W - r0) - wr : 0, ncol = min(rr, W - c0) - wc;
      double2* Ck = C + k * (int64_t)W * W + (int64_t)(r0 + wr) * W + c0 + wc;
      unsigned mx = 0u;
      for (int gi = 0; gi * GROUP < nch; ++gi, ++G) {
        ok = mbar_wait(&acc_full, (uint32_t)G & 1u);
        ok = __all_sync(0xffffffffu, ok && !abort_sh);   // tcgen05.ld is warp-collective
        if (!ok) break;
        tc_fence_after();
        const bool add = accum || gi > 0, final_group = (gi + 1) * GROUP >= nch;
#pragma unroll 1
        for (int s0 = half * SLAB; s0 < DRAIN_COLS; s0 += 2 * SLAB) {
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            uint32_t x[NLEV][4];
#pragma unroll
            for (int l = 0; l < NLEV; ++l) tmem_ld4_async(lane_addr + (uint32_t)(l * NCP + s0 + 4 * b), x[l]);
#pragma unroll
            for (int l = 0; l < NLEV; ++l) tmem_wait_ld4(x[l]);
            if (b == 1 && s0 + 2 * SLAB >= DRAIN_COLS) {   // the thread's last TMEM read of this drain
              tc_fence_before();
              mbar_arrive(&acc_empty);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              int I[NLEV];
#pragma unroll
              for (int l = 0; l < NLEV; ++l) I[l] = __float2int_rn(__uint_as_float(x[l][j]));
              // sum_l I_l 2^(41 - 8 l), the levels 6 and 7 rounded to the unit 2^-55
              const long long hi = (long long)I[0] * 65536 + ((long long)I[1] * 256 + I[2]);
              const long long lo = (long long)I[3] * 65536 + ((long long)I[4] * 256 + I[5]);
              const long long v = (hi << 25) + (lo << 1) + (((long long)I[6] * 256 + (I[7] + 16384)) >> 15);
              mine[2 * (4 * b + j)] = bad ? __longlong_as_double(0x7FF8000000000000ll) : scaled_double(v, es);
            }
          }
          __syncwarp();
          // the slab to global memory, 8 columns (128 bytes) of a row by 8 lanes
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (4 * q < nrow && s0 < ncol) {
              double2* dst = Ck + (int64_t)(4 * q) * W + s0;
              double2 v = slab[(wr + 4 * q) * (SLAB + 1) + wc];
              if (add) {
                const double2 o = *dst;
                v.x += o.x;
                v.y += o.y;
              }
              *dst = v;
              if (final_group) mx = max(mx, (unsigned)(max(mag_bits(v.x), mag_bits(v.y)) >> 32));
            }
          __syncwarp();
        }
      }
      if (ec && ok) {
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const int ex = (int)(mx >> 20);
        if (lane == 0 && (P == 1 || k1 < n)) atomicMax(&ec[k], ex == 0x7FF ? ZEXP_BAD : ex - 1022);
      }
    }
    if (!ok) {
      atomicOr(&st->bits, ST_TIMEOUT);
      abort_sh = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
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
  // matrices per tile: an unshared tile of W = 32 leaves half of the MMA rows empty and its chunks, loads and
  // drain take their latencies alone (gradient at W = 32, 9,216 k-points: adjoint 7.2 ms, two to a tile 5.3)
  const int P = W <= 16 ? 4 : W <= 32 ? 2 : 1;
  const int ncp = rr <= 32 || rr > 48 ? 64 : 48;
  const size_t sm = (size_t)ND * A_SLICE + (size_t)ND * ncp * ROW_BYTES +
                    ((size_t)2 * CH * RAW_PITCH + EPI_THREADS / 2 * (SLAB + 1)) * sizeof(double2) + 1024;
  int dev = 0, nsm = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    if (ec) {
      e = cudaMemsetAsync(ec, 0xC0, sizeof(int) * (size_t)n, s);   // a large negative exponent
      if (e != cudaSuccess) return e;
    }
    const int64_t tiles = ((int64_t)n + P - 1) / P * nt * nt;
    kern<<<(int)std::min<int64_t>(tiles, std::max(nsm, 1)), THREADS, sm, s>>>(A, B, C, ec, W, n, nt, rr,
                                                                              upper ? 1 : 0, accum ? 1 : 0, st);
    return cudaGetLastError();
  };
  if (P == 4) return go(zgemm_tc64_kernel<64, 4>);
  if (P == 2) return go(zgemm_tc64_kernel<64, 2>);
  return ncp == 48 ? go(zgemm_tc64_kernel<48, 1>) : go(zgemm_tc64_kernel<64, 1>);
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
