// Step (1) of List 1/2 in FP64 grade on the 5th-generation tensor cores.
//
// The dense contraction C[n_k x 3W^2] = Coef[n_k x N_R] . Basis[N_R x 3W^2] of k_fourier_tc.cu
// with seven fixed-point slices per operand instead of four: every coefficient (|c| <= 1) and
// every basis entry (scaled by 2^-e_n, e_n the exponent of its column's largest magnitude) is
// rounded to 55 fractional bits and cut into signed base-256 digits,
//   x = sum_{i<7} s_i 2^(-7-8i),  |s_i| <= 128, exact in BF16,
// and the 28 digit products of the levels l = i + j <= 6 are kept.  A level sum over 128 of K is
// an integer of at most 7 x 128 x 2^14 < 2^24, exact in the FP32 accumulator; the epilogue adds
// the levels exactly in two int64 per output and rounds to FP64 once.  The error is the operand
// rounding (2^-56 of the operand scales) and the dropped levels (2^-57.6 r.m.s. per product),
// about 2^-51 of the result at N_R = 1331, where a chain of 2 N_h FP64 multiply-adds leaves
// about 2^-48 (relative 2-norm errors against an exact sum are in the tests).
//
// What bounds it: the FP64 pipe issues one warp instruction in 16 cycles, so the FMA form
// (k_fourier.cu, 95 % of that pipe) takes 6 N_R W^2 / 1.2 TFLOP/s; here the 28 BF16 products of
// an output run at the tensor rate.  The A operand is read from L2 once per 32 columns
// and the kernel takes in 143 KB per 64-wide K block of a tile.
//
//   basis_exp7 / basis_slice7   once per call: column exponents, Bt[7][Npad][Kp] (K-major bf16)
//   coef_slice7                 per batch: FP64 phases (exact integer argument reduction), A[7][Mpad][Kp]
//   fourier_tc64                per batch: persistent tcgen05 GEMM, 128 x 32 output tiles
//
// Every mbarrier wait is bounded; on timeout the CTA records ST_TIMEOUT, drains its own copies
// (bounded), frees its TMEM and returns.
#include <algorithm>
#include <climits>

#include <cuda.h>
#include <cuda_bf16.h>

#include "digits.cuh"
#include "kubo_internal.cuh"
#include "tc_ptx.cuh"

namespace kubo {

namespace {

using namespace tc;
using namespace dig;

constexpr int BM = 128;          // k-points per tile (UMMA M)
constexpr int BN = 32;           // output columns per tile: 7 levels x 32 columns x 2 sets of TMEM
constexpr int BK = 64;           // K per block: one 128-byte swizzle row of bf16
constexpr int NS = ND;           // seven slices per operand and levels kept: 28 digit products
constexpr int NACC = 2;          // accumulator sets: one drained while the other is filled
constexpr int SET_COLS = 256;    // TMEM columns of a set (7 x 32 used)
constexpr int DRAIN = 2;         // K blocks per drain: 7 x 128 x 2^14 < 2^24
constexpr int TILE_A = BM * BK * 2;        // 16 KB, one slice
constexpr int TILE_B = BN * BK * 2;        // 4 KB, one slice; a block's seven are stacked
constexpr int NB = 2;                      // B blocks in flight
// A slices in flight.  Slice i of a block is read by one group of MMAs (against the stacked B
// slices 0 .. 6 - i) and its slot is free again, so the ring turns over slice by slice; a whole
// block per stage (140 KB) would leave room for one stage.
constexpr int NA = 10;
constexpr int SMEM_BYTES = NA * TILE_A + NB * NS * TILE_B + 1024;
constexpr int TC_THREADS = 320;            // TMA warp, MMA warp, 8 epilogue warps
constexpr int EPI_THREADS = TC_THREADS - 64;
constexpr int EPI_COLS = BN / 2;           // columns per epilogue thread
constexpr int TMEM_COLS = 512;
constexpr int EXP_NONFINITE = INT_MAX;     // column with an infinite or NaN basis entry

__host__ __device__ constexpr uint32_t idesc_n(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// ------------------------------------------------------------------ operand preparation
// e[a W^2 + q] (a = H, d_x, d_y; padding columns 0): exponent with |basis| < 2^e over K, from the
// bit patterns.  Block: 32 columns q x 8 slices of the half set.
__global__ void __launch_bounds__(256) basis_exp7_kernel(const double* __restrict__ Bp,
                                                         const int* __restrict__ Rh, int N_h,
                                                         int WW, int Npad, int* __restrict__ e) {
  __shared__ unsigned long long red[3][8][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int q = blockIdx.x * 32 + x;
  unsigned long long m[3] = {0ull, 0ull, 0ull};
  if (q < WW) {
    if (y == 0) m[0] = mag_bits(Bp[q]);
    for (int h = y; h < N_h; h += 8) {
      const double a = Bp[(size_t)(1 + 2 * h) * WW + q], b = Bp[(size_t)(2 + 2 * h) * WW + q];
      const unsigned long long ab = max(mag_bits(a), mag_bits(b));
      const double big = __longlong_as_double((long long)ab);
      m[0] = max(m[0], ab);
      m[1] = max(m[1], mag_bits((double)Rh[3 * h] * big));
      m[2] = max(m[2], mag_bits((double)Rh[3 * h + 1] * big));
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) red[a][y][x] = m[a];
  __syncthreads();
  if (y < 3 && q < WW) {
    unsigned long long v = 0ull;
    for (int i = 0; i < 8; ++i) v = max(v, red[y][i][x]);
    const int ex = (int)(v >> 52);
    // |x| < 2^(ex - 1022); a subnormal maximum takes the exponent of the smallest normal
    e[y * WW + q] = ex == 0x7FF ? EXP_NONFINITE : (v == 0ull ? 0 : (ex == 0 ? -1021 : ex - 1022));
  }
  if (blockIdx.x == 0)
    for (int n = 3 * WW + threadIdx.x; n < Npad; n += 256) e[n] = 0;
}

// Bt[s][n][k]: block = 32 columns q x 32 vectors h (64 of K), A_h and B_h read once (rows
// coalesced over q) and transposed through shared memory for the three column groups.
__global__ void __launch_bounds__(256) basis_slice7_kernel(const double* __restrict__ Bp,
                                                           const int* __restrict__ Rh,
                                                           const int* __restrict__ e, int N_h,
                                                           int WW, int Npad, int Kp,
                                                           __nv_bfloat16* __restrict__ Bt) {
  __shared__ double sA[32][33], sB[32][33];
  const int q0 = blockIdx.x * 32, h0 = blockIdx.y * 32;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int hh = y; hh < 32; hh += 8) {
    const int h = h0 + hh, q = q0 + x;
    double a = 0.0, b = 0.0;
    if (q < WW && h < N_h) {
      a = Bp[(size_t)(1 + 2 * h) * WW + q];
      b = Bp[(size_t)(2 + 2 * h) * WW + q];
    } else if (q < WW && h == N_h) {
      a = Bp[q];   // the R = 0 row, against the constant column 2 N_h
    }
    sA[hh][x] = a;
    sB[hh][x] = b;
  }
  __syncthreads();
  const size_t plane = (size_t)Npad * Kp;
  const int h = h0 + x;
  const double rx = h < N_h ? (double)Rh[3 * h] : 0.0, ry = h < N_h ? (double)Rh[3 * h + 1] : 0.0;
  if (2 * h >= Kp) return;
  for (int qq = y; qq < 32; qq += 8) {
    const int q = q0 + qq;
    if (q >= WW) break;
    const double a = sA[x][qq], b = sB[x][qq];
#pragma unroll
    for (int al = 0; al < 3; ++al) {
      const int n = al * WW + q;
      const double r = al == 1 ? rx : ry;
      const double vc = al == 0 ? a : r * b, vs = al == 0 ? b : -r * a;
      const int en = e[n];
      uint32_t dc[NS], ds[NS];
      digits7(fixed55(vc, en == EXP_NONFINITE ? 1024 : en), dc);
      digits7(fixed55(vs, en == EXP_NONFINITE ? 1024 : en), ds);
#pragma unroll
      for (int i = 0; i < NS; ++i)
        *reinterpret_cast<uint32_t*>(Bt + i * plane + (size_t)n * Kp + 2 * h) = bf16_pair(dc[i], ds[i]);
    }
  }
}

// padding columns n >= 3 W^2 of Bt
__global__ void basis_pad7_kernel(int n0, int Npad, int Kp, __nv_bfloat16* __restrict__ Bt) {
  const size_t plane = (size_t)Npad * Kp;
  const size_t cnt = (size_t)(Npad - n0) * Kp / 2;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < cnt * NS;
       t += (size_t)gridDim.x * blockDim.x)
    reinterpret_cast<uint32_t*>(Bt + (t / cnt) * plane + (size_t)n0 * Kp)[t % cnt] = 0u;
}

// A[s][m][k] for m < Mpad (rows >= n zero), k < Kp: the phases are those of mesh_phase (FP64
// products of the three twiddles), rounded to 55 fractional bits.
__global__ void __launch_bounds__(256) coef_slice7_kernel(Model md, Mesh mesh, KList kl, int Mpad,
                                                          int Kp, __nv_bfloat16* __restrict__ A) {
  const int npair = Kp / 2;
  const size_t plane = (size_t)Mpad * Kp;
  const FastDiv f1((uint32_t)mesh.N1), f2((uint32_t)mesh.N2), f3((uint32_t)mesh.N3);
  const int64_t total = (int64_t)Mpad * npair;
  const FastDiv fp((uint32_t)npair);
  for (int64_t i0 = (int64_t)blockIdx.x * 256; i0 < total; i0 += (int64_t)gridDim.x * 256) {
    const int64_t idx = i0 + threadIdx.x;
    if (idx >= total) break;
    int m, h;   // (idx npair is beyond 2^32 from some 10,000 rows at N_R = 1331)
    if (idx < 0x100000000ll) {
      uint32_t rem;
      m = (int)fp.divmod((uint32_t)idx, rem);
      h = (int)rem;
    } else {
      m = (int)(idx / npair);
      h = (int)(idx - (int64_t)m * npair);
    }
    uint32_t dc[NS], ds[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) dc[i] = ds[i] = 0u;
    if (m < kl.n) {
      if (h < md.N_h) {
        int j1, j2, j3;
        mesh_coords(mesh, klist_get(kl, m), j1, j2, j3);
        const int* r = md.Rh + 3 * h;
        const double2 p = cmul(md.tab[md.tab_off[0] + posmod((long long)j1 * r[0], f1)],
                               md.tab[md.tab_off[1] + posmod((long long)j2 * r[1], f2)]);
        const double2 c = cmul(p, md.tab[md.tab_off[2] + posmod((long long)j3 * r[2], f3)]);
        // |c| exceeds 1 by an ulp at most: |q| <= 2^55 + 2^3, the top digit still 128
        digits7(fixed55(c.x, 0), dc);
        digits7(fixed55(c.y, 0), ds);
      } else if (h == md.N_h) {
        dc[0] = __float_as_uint(128.0f);   // 1: the R = 0 term
      }
    }
    const size_t o = (size_t)m * Kp + 2 * h;
#pragma unroll
    for (int i = 0; i < NS; ++i) *reinterpret_cast<uint32_t*>(A + i * plane + o) = bf16_pair(dc[i], ds[i]);
  }
}

// ------------------------------------------------------------------ transposed sum (gradient)
// G_rows[1 + 2 N_h][3 W^2] += Coef^T . [Hbar | dxHbar | dyHbar]: the same GEMM with the k-points as its
// inner index.  A[s][row][k]: rows 1, cos k.R_h, sin k.R_h (grad_finalize_kernel's order), zero for
// k >= n.
__global__ void __launch_bounds__(256) coef_t_slice7_kernel(Model md, Mesh mesh, KList kl, int Mpad,
                                                            int Kp, __nv_bfloat16* __restrict__ A) {
  const int npair = Kp / 2;
  const size_t plane = (size_t)Mpad * Kp;
  const FastDiv f1((uint32_t)mesh.N1), f2((uint32_t)mesh.N2), f3((uint32_t)mesh.N3);
  const int64_t total = (int64_t)(md.N_h + 1) * npair;
  for (int64_t idx = blockIdx.x * (int64_t)256 + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * 256) {
    const int h = (int)(idx / npair) - 1;
    const int k2 = 2 * (int)(idx % npair);
    uint32_t dc[2][NS], ds[2][NS];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
#pragma unroll
      for (int i = 0; i < NS; ++i) dc[b][i] = ds[b][i] = 0u;
      if (k2 + b >= kl.n) continue;
      if (h < 0) {
        dc[b][0] = __float_as_uint(128.0f);
      } else {
        int j1, j2, j3;
        mesh_coords(mesh, klist_get(kl, k2 + b), j1, j2, j3);
        const int* r = md.Rh + 3 * h;
        const double2 p = cmul(md.tab[md.tab_off[0] + posmod((long long)j1 * r[0], f1)],
                               md.tab[md.tab_off[1] + posmod((long long)j2 * r[1], f2)]);
        const double2 c = cmul(p, md.tab[md.tab_off[2] + posmod((long long)j3 * r[2], f3)]);
        digits7(fixed55(c.x, 0), dc[b]);
        digits7(fixed55(c.y, 0), ds[b]);
      }
    }
    __nv_bfloat16* rc = A + (size_t)(1 + h) * Kp + k2;
    __nv_bfloat16* rs = A + (size_t)(1 + md.N_h + h) * Kp + k2;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      *reinterpret_cast<uint32_t*>(rc + i * plane) = bf16_pair(dc[0][i], dc[1][i]);
      if (h >= 0) *reinterpret_cast<uint32_t*>(rs + i * plane) = bf16_pair(ds[0][i], ds[1][i]);
    }
  }
}

// e[c]: exponent above column c of M [n][N] (rows blockIdx.y * 256 ..; e starts far below zero)
__global__ void __launch_bounds__(256) col_exp7_kernel(const double* __restrict__ M, int n, int N,
                                                       int* __restrict__ e) {
  __shared__ unsigned red[8][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + x;
  unsigned m = 0u;
  if (c < N)
    for (int k = blockIdx.y * 256 + y; k < min(n, (int)blockIdx.y * 256 + 256); k += 8)
      m = max(m, (unsigned)(mag_bits(M[(size_t)k * N + c]) >> 32));
  red[y][x] = m;
  __syncthreads();
  if (y == 0 && c < N) {
    for (int i = 1; i < 8; ++i) m = max(m, red[i][x]);
    const int ex = (int)(m >> 20);
    atomicMax(&e[c], ex == 0x7FF ? EXP_NONFINITE : ex - 1022);
  }
}

// Bt[s][c][k] of M [n][N]: 32 columns x 64 k per block, transposed through shared memory
__global__ void __launch_bounds__(256) col_slice7_kernel(const double* __restrict__ M, int n, int N,
                                                         const int* __restrict__ e, int Npad, int Kp,
                                                         __nv_bfloat16* __restrict__ Bt) {
  __shared__ double sm[64][33];
  const int c0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int kk = y; kk < 64; kk += 8) {
    const int k = k0 + kk, c = c0 + x;
    sm[kk][x] = k < n && c < N ? M[(size_t)k * N + c] : 0.0;
  }
  __syncthreads();
  const size_t plane = (size_t)Npad * Kp;
  for (int cc = y; cc < 32; cc += 8) {
    const int c = c0 + cc;
    if (c >= N) break;
    const int ec = e[c] == EXP_NONFINITE ? 1024 : e[c];
    uint32_t d0[NS], d1[NS];
    digits7(fixed55(sm[2 * x][cc], ec), d0);
    digits7(fixed55(sm[2 * x + 1][cc], ec), d1);
#pragma unroll
    for (int i = 0; i < NS; ++i)
      *reinterpret_cast<uint32_t*>(Bt + i * plane + (size_t)c * Kp + k0 + 2 * x) = bf16_pair(d0[i], d1[i]);
  }
}

// ------------------------------------------------------------------ the tcgen05 GEMM
// Persistent: CTA b walks tiles b, b + gridDim.x, ...; group_m M tiles per column tile in a row,
// so a B tile serves several tiles and the group's A slices stay in L2.
__global__ void __launch_bounds__(TC_THREADS, 1)
    fourier_tc64_kernel(const __grid_constant__ CUtensorMap mapA,
                        const __grid_constant__ CUtensorMap mapB, const int* __restrict__ col_exp,
                        int Mpad, int Npad, int nkb, int n_rows, int WW, double* Hp, double* Xp,
                        double* Yp, int64_t ldo, bool accum, DevStatus* st, int group_m,
                        bool vec) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t a_full[NA], a_empty[NA], b_full[NB], b_empty[NB];
  __shared__ __align__(8) uint64_t acc_full[NACC], acc_empty[NACC], done_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_mt = Mpad / BM, n_nt = Npad / BN, n_tiles = n_mt * n_nt;
  const int groups_per_tile = (nkb + DRAIN - 1) / DRAIN;
  auto tile_origin = [&](int id, int& m0, int& n0) {
    const int per_group = group_m * n_nt;
    const int grp = id / per_group;
    const int gm0 = grp * group_m;
    const int gsz = min(group_m, n_mt - gm0);
    const int in = id - grp * per_group;
    n0 = (in / gsz) * BN;
    m0 = (gm0 + in % gsz) * BM;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < NA; ++s) { mbar_init(&a_full[s], 1); mbar_init(&a_empty[s], 1); }
    for (int s = 0; s < NB; ++s) { mbar_init(&b_full[s], 1); mbar_init(&b_empty[s], 1); }
    for (int a = 0; a < NACC; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], EPI_THREADS);
    }
    mbar_init(&done_bar, 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
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
  auto bufA = [&](int s) { return base + (size_t)s * TILE_A; };
  auto bufB = [&](int s) { return base + (size_t)NA * TILE_A + (size_t)s * NS * TILE_B; };

  if (warp == 0) {
    // ---------------- TMA producer: g counts K blocks, u A slices, over all tiles of the CTA
    if (lane == 0) {
      int g = 0, u = 0;
      bool ok = true;
      for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
        int m0, n0;
        tile_origin(id, m0, n0);
        for (int kb = 0; kb < nkb && ok; ++kb) {
          const int sb = g % NB;
          if (abort_sh || (g >= NB && !mbar_wait(&b_empty[sb], ((uint32_t)(g / NB) & 1u) ^ 1u))) {
            ok = false;
            break;
          }
          mbar_expect_tx(&b_full[sb], NS * TILE_B);
          for (int j = 0; j < NS; ++j)
            tma_load_2d(bufB(sb) + j * TILE_B, &mapB, &b_full[sb], kb * BK, j * Npad + n0);
          ++g;
          for (int i = 0; i < NS; ++i) {
            const int sa = u % NA;
            if (abort_sh || (u >= NA && !mbar_wait(&a_empty[sa], ((uint32_t)(u / NA) & 1u) ^ 1u))) {
              ok = false;
              break;
            }
            mbar_expect_tx(&a_full[sa], TILE_A);
            tma_load_2d(bufA(sa), &mapA, &a_full[sa], kb * BK, i * Mpad + m0);
            ++u;
          }
        }
      }
      if (!ok) {
        atomicOr(&st->bits, ST_TIMEOUT);
        abort_sh = 1;
      }
      // every issued copy must have landed before the CTA may exit
      for (int q = (g > NB ? g - NB : 0); q < g; ++q) mbar_wait(&b_full[q % NB], (uint32_t)(q / NB) & 1u);
      for (int q = (u > NA ? u - NA : 0); q < u; ++q) mbar_wait(&a_full[q % NA], (uint32_t)(q / NA) & 1u);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer.  Slice A_i against the stacked B slices 0 .. 6 - i (rows j BN ..
    // of one swizzled K-major operand): accumulator columns of the levels i .. 6.  A_0 comes
    // first and initialises every level of a drain group.
    if (lane == 0) {
      int g = 0, u = 0, G = 0;
      bool ok = true;
      for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
        for (int kb = 0; kb < nkb && ok; ++kb, ++g) {
          const int sb = g % NB, a = G % NACC;
          const bool first = kb % DRAIN == 0;
          const bool last = kb % DRAIN == DRAIN - 1 || kb == nkb - 1;
          if (abort_sh || (first && G >= NACC && !mbar_wait(&acc_empty[a], (uint32_t)(G / NACC - 1) & 1u)) ||
              !mbar_wait(&b_full[sb], (uint32_t)(g / NB) & 1u)) {
            ok = false;
            break;
          }
#pragma unroll
          for (int i = 0; i < NS; ++i) {
            const int sa = u % NA;
            if (!mbar_wait(&a_full[sa], (uint32_t)(u / NA) & 1u)) {
              ok = false;
              break;
            }
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
              const uint64_t da = umma_desc_sw128(smem_u32(bufA(sa)) + kk * 32);
              const uint64_t db = umma_desc_sw128(smem_u32(bufB(sb)) + kk * 32);
              umma_bf16(tmem + (uint32_t)(a * SET_COLS + i * BN), da, db, idesc_n((NS - i) * BN),
                        (i > 0 || !first || kk > 0) ? 1u : 0u);
            }
            umma_commit(&a_empty[sa]);
            ++u;
          }
          if (!ok) break;
          umma_commit(&b_empty[sb]);
          if (last) {
            umma_commit(&acc_full[a]);
            ++G;
          }
        }
      }
      if (!ok) {
        atomicOr(&st->bits, ST_TIMEOUT);
        abort_sh = 1;
      }
      umma_commit(&done_bar);   // all issued MMAs complete
    }
  } else {
    // ---------------- epilogue: warp w owns TMEM lanes 32 (w % 4) .. + 31 and half the columns
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const int c_lo = ((warp - 2) >> 2) * EPI_COLS;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c_lo;
    bool ok = true;
    int G = 0;
    for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
      int m0, n0;
      tile_origin(id, m0, n0);
      // levels 0-2 and 3-6 of an output: sum_l I_l 2^(16 - 8 l) and sum_l I_l 2^(48 - 8 l), each
      // exact (a level sum is below 2^24, so a drain adds less than 2^41 and 2^49)
      long long hi[EPI_COLS], lo[EPI_COLS];
#pragma unroll
      for (int j = 0; j < EPI_COLS; ++j) hi[j] = lo[j] = 0;
      for (int gi = 0; gi < groups_per_tile; ++gi, ++G) {
        const int a = G % NACC;
        ok = mbar_wait(&acc_full[a], (uint32_t)(G / NACC) & 1u);
        ok = __all_sync(0xffffffffu, ok && !abort_sh);   // tcgen05.ld is warp-collective
        if (!ok) break;
        tc_fence_after();
        uint32_t rb[2][16];
        const uint32_t set_addr = lane_addr + (uint32_t)(a * SET_COLS);
        tmem_ld16_async(set_addr, rb[0]);
        tmem_wait_ld16(rb[0]);
#pragma unroll
        for (int l = 0; l < NS; ++l) {
          if (l + 1 < NS) tmem_ld16_async(set_addr + (uint32_t)((l + 1) * BN), rb[(l + 1) & 1]);
          const int w = l < 3 ? 1 << (16 - 8 * l) : 1 << (48 - 8 * l);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int v = __float2int_rn(__uint_as_float(rb[l & 1][j]));
            if (l < 3) hi[j] += (long long)v * w;
            else lo[j] += (long long)v * w;
          }
          if (l + 1 < NS) tmem_wait_ld16(rb[(l + 1) & 1]);
        }
        tc_fence_before();
        mbar_arrive(&acc_empty[a]);
      }
      if (!ok) break;
      const int64_t grow = m0 + row;
      if (grow < n_rows) {
        // C = 2^e (hi 2^-30 + lo 2^-62): both parts are exact in FP64, the FMA rounds once
        const int n1 = n0 + c_lo;
        const int* ce = col_exp + n1;
        double v[EPI_COLS];
#pragma unroll
        for (int j = 0; j < EPI_COLS; ++j) {
          const int e = ce[j], ex = e - 30;
          const double s = fma((double)lo[j], 0x1p-32, (double)hi[j]);
          if (ex >= -900 && ex <= 900) v[j] = s * __longlong_as_double((long long)(1023 + ex) << 52);
          else v[j] = e == EXP_NONFINITE ? __longlong_as_double(0x7FF8000000000000ll) : ldexp(s, ex);
        }
        // column n is entry n mod W^2 of H, d_x H or d_y H (n / W^2); a thread's columns lie in
        // one of them when W^2 is a multiple of 16 (vec: and the outputs are 16-byte aligned)
        if (vec) {
          if (n1 < 3 * WW) {
            const int a = n1 / WW;
            double* dst = (a == 0 ? Hp : a == 1 ? Xp : Yp) + grow * ldo + (n1 - a * WW);
#pragma unroll
            for (int j = 0; j < EPI_COLS; j += 2) {
              double2 w = make_double2(v[j], v[j + 1]);
              if (accum) {
                const double2 o = *reinterpret_cast<const double2*>(dst + j);
                w.x += o.x;
                w.y += o.y;
              }
              *reinterpret_cast<double2*>(dst + j) = w;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < EPI_COLS; ++j) {
            const int n = n1 + j;
            if (n < 3 * WW) {
              const int a = n < WW ? 0 : n < 2 * WW ? 1 : 2;
              double* dst = (a == 0 ? Hp : a == 1 ? Xp : Yp) + grow * ldo + (n - a * WW);
              *dst = accum ? *dst + v[j] : v[j];
            }
          }
        }
      }
    }
    if (!ok) {
      atomicOr(&st->bits, ST_TIMEOUT);
      abort_sh = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (lane == 0) mbar_wait(&done_bar, 0);   // no MMA may still be writing TMEM
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

}  // namespace

int tc64_pad_n(int W) { return (3 * W * W + BN - 1) / BN * BN; }
int tc64_slices() { return NS; }

cudaError_t launch_basis_split64(const double* Bp, const int* Rh, int N_h, int W, int Npad, int Kp,
                                 int* col_exp, void* Bt, cudaStream_t s) {
  const int WW = W * W;
  const int gq = (WW + 31) / 32;
  basis_exp7_kernel<<<gq, 256, 0, s>>>(Bp, Rh, N_h, WW, Npad, col_exp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  basis_slice7_kernel<<<dim3(gq, Kp / 64), 256, 0, s>>>(Bp, Rh, col_exp, N_h, WW, Npad, Kp,
                                                        (__nv_bfloat16*)Bt);
  e = cudaGetLastError();
  if (e != cudaSuccess || 3 * WW == Npad) return e;
  basis_pad7_kernel<<<64, 256, 0, s>>>(3 * WW, Npad, Kp, (__nv_bfloat16*)Bt);
  return cudaGetLastError();
}

cudaError_t launch_coef_split64(const Model& md, const Mesh& mesh, const KList& kl, int Mpad,
                                int Kp, void* A, cudaStream_t s) {
  const int64_t total = (int64_t)Mpad * (Kp / 2);
  const int grid = (int)std::min<int64_t>((total + 255) / 256, 152 * 32);
  coef_slice7_kernel<<<grid, 256, 0, s>>>(md, mesh, kl, Mpad, Kp, (__nv_bfloat16*)A);
  return cudaGetLastError();
}

// out: three arrays [n_rows][W^2] of row stride ldo, overwritten or added to
static cudaError_t launch_gemm7(const void* A, const void* Bt, const int* col_exp, int Mpad, int Npad,
                                int Kp, int n_rows, int W, double* Hp, double* Xp, double* Yp,
                                int64_t ldo, bool accum, DevStatus* st, cudaStream_t s) {
  if (n_rows <= 0) return cudaSuccess;
  if (Mpad % BM || Npad % BN || Kp % BK) return cudaErrorInvalidValue;
  CUtensorMap mA, mB;
  if (!tc_encode_bf16(&mA, A, (uint64_t)Kp, (uint64_t)NS * Mpad, BK, BM) ||
      !tc_encode_bf16(&mB, Bt, (uint64_t)Kp, (uint64_t)NS * Npad, BK, BN))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(fourier_tc64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       SMEM_BYTES);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // M tiles rasterised together: the group's A slices (128 x Kp x 14 bytes per M tile) within
  // 48 MB of the L2, so that the basis is read from HBM once per group
  const int64_t per_m = (int64_t)BM * Kp * 2 * NS;
  const int group_m = (int)std::max<int64_t>(1, std::min<int64_t>(64, ((int64_t)48 << 20) / per_m));
  const bool vec = W % 4 == 0 && ldo % 2 == 0 && (((uintptr_t)Hp | (uintptr_t)Xp | (uintptr_t)Yp) & 15) == 0;
  const int tiles = (Mpad / BM) * (Npad / BN);
  fourier_tc64_kernel<<<std::min(tiles, std::max(nsm, 1)), TC_THREADS, SMEM_BYTES, s>>>(
      mA, mB, col_exp, Mpad, Npad, Kp / BK, n_rows, W * W, Hp, Xp, Yp, ldo, accum, st, group_m, vec);
  return cudaGetLastError();
}

cudaError_t launch_fourier_tc64(const void* A, const void* Bt, const int* col_exp, int Mpad,
                                int Npad, int Kp, int n_rows, int W, double* Hp, double* Xp,
                                double* Yp, DevStatus* st, cudaStream_t s) {
  return launch_gemm7(A, Bt, col_exp, Mpad, Npad, Kp, n_rows, W, Hp, Xp, Yp, (int64_t)W * W, false, st, s);
}

cudaError_t launch_grad_fourier_t(const Model& md, const Mesh& mesh, const KList& kl, const double* Mbar,
                                  void* A, void* Bt, int* col_exp, double* Gacc, DevStatus* st,
                                  cudaStream_t s) {
  if (kl.n <= 0) return cudaSuccess;
  const int WW = md.W * md.W, N = 3 * WW, rows = 1 + 2 * md.N_h;
  const int Npad = tc64_pad_n(md.W), Mpad = tc_pad_m(rows), Kp = tc_pad_k(kl.n);
  const int64_t total = (int64_t)(md.N_h + 1) * (Kp / 2);
  coef_t_slice7_kernel<<<(int)std::min<int64_t>((total + 255) / 256, 152 * 32), 256, 0, s>>>(
      md, mesh, kl, Mpad, Kp, (__nv_bfloat16*)A);
  cudaError_t e = cudaMemsetAsync(col_exp, 0xC0, sizeof(int) * (size_t)Npad, s);
  if (e != cudaSuccess) return e;
  col_exp7_kernel<<<dim3((N + 31) / 32, (kl.n + 255) / 256), 256, 0, s>>>(Mbar, kl.n, N, col_exp);
  col_slice7_kernel<<<dim3((N + 31) / 32, Kp / 64), 256, 0, s>>>(Mbar, kl.n, N, col_exp, Npad, Kp,
                                                                  (__nv_bfloat16*)Bt);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_gemm7(A, Bt, col_exp, Mpad, Npad, Kp, rows, md.W, Gacc, Gacc + WW, Gacc + 2 * WW, N, true,
                      st, s);
}

}  // namespace kubo
