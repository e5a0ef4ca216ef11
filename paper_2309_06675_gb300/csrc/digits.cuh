// Signed base-256 digits in BF16 or FP16 for exact tensor-core products (k_fourier_tc64.cu, k_zgemm_tc64.cu):
// x 2^-e = sum_{i<7} s_i 2^(-7-8i) + O(2^-56), |s_i| <= 128, for |x| < 2^e.
#pragma once

#include <stdint.h>

namespace kubo {
namespace dig {

constexpr int ND = 7;   // digits per number: 55 fractional bits

// round(x 2^(55 - e)) for |x| <= 2^e, from the FP64 bit pattern (round half up of the
// magnitude; no FP64 instruction): |q| <= 2^55
__device__ __forceinline__ long long fixed55(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & ((1ull << 52) - 1);
  if (ex == 0) ex = 1;
  else m |= 1ull << 52;
  const int sh = 1020 + e - ex;   // x 2^(55-e) = m 2^(ex - 1075 + 55 - e) = m 2^-sh, sh >= -3
  const unsigned long long q = sh <= 0 ? m << -sh : (sh < 64 ? (m + (1ull << (sh - 1))) >> sh : 0ull);
  return (b >> 63) ? -(long long)q : (long long)q;
}
// digits of q (|q| <= 2^55), most significant first, as FP32 integers: adding 128 to the six
// low digits makes them plain bytes; a byte b becomes the float b - 128 by placing it in the
// mantissa of 2^23 and subtracting 2^23 + 128 (exact).  The upper half of such a float is the
// digit in BF16.
__device__ __forceinline__ void digits7(long long q, uint32_t (&d)[ND]) {
  const long long v = q + 0x0000808080808080ll;
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)((unsigned long long)v >> 32);
#pragma unroll
  for (int j = 0; j < 6; ++j) {   // byte j of v -> digit 6 - j
    const uint32_t f = __byte_perm(j < 4 ? lo : hi, 0x4B000000u, 0x7650u | (j & 3));
    d[6 - j] = __float_as_uint(__uint_as_float(f) - 8388736.0f);
  }
  d[0] = __float_as_uint((float)(int)(v >> 48));
}
// two digits as a bf16 pair (a low)
__device__ __forceinline__ uint32_t bf16_pair(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x7632); }

// The same digits of two numbers as FP16 pairs (q1 low): a byte b becomes b - 128 by placing it in the
// mantissa of 1024 and subtracting 1152 (exact); 11 byte permutes for both numbers where the BF16 form
// takes 23 integer instructions.
__device__ __forceinline__ uint32_t h2_sub(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ void digits7_h2(long long q1, long long q2, uint32_t (&d)[ND]) {
  const long long v1 = q1 + 0x0080808080808080ll, v2 = q2 + 0x0080808080808080ll;
  const uint32_t l1 = (uint32_t)v1, l2 = (uint32_t)v2;
  const uint32_t h1 = (uint32_t)((unsigned long long)v1 >> 32), h2 = (uint32_t)((unsigned long long)v2 >> 32);
  constexpr uint32_t K = 0x64646464u, C = 0x64806480u;   // 1024's high byte; 1152
  const uint32_t t01 = __byte_perm(l1, l2, 0x5140), t23 = __byte_perm(l1, l2, 0x7362);
  const uint32_t t45 = __byte_perm(h1, h2, 0x5140), t6 = __byte_perm(h1, h2, 0x7632);
  d[6] = h2_sub(__byte_perm(t01, K, 0x4140), C);
  d[5] = h2_sub(__byte_perm(t01, K, 0x4342), C);
  d[4] = h2_sub(__byte_perm(t23, K, 0x4140), C);
  d[3] = h2_sub(__byte_perm(t23, K, 0x4342), C);
  d[2] = h2_sub(__byte_perm(t45, K, 0x4140), C);
  d[1] = h2_sub(__byte_perm(t45, K, 0x4342), C);
  d[0] = h2_sub(t6 + 0x64006400u, C);   // the biased top digit, 0 .. 256
}

}  // namespace dig
}  // namespace kubo
