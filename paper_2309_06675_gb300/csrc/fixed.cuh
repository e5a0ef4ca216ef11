// Fixed-point arithmetic of FP64 grade on the integer pipe.
//
// GB300 issues an FP64 multiply-add for 2 lanes per SM clock and a 32 x 32 + 64-bit integer
// multiply-add (IMAD.WIDE) for 32 (both measured), so a product of two 59-bit fixed-point numbers by
// three integer multiply-adds runs five times as fast as an FP64 one.  A number |x| < 1 is
// X = round(x 2^59), held as two signed limbs, X = h 2^28 + l with |h| < 2^31 and |l| <= 2^27;
//   X Y = hh 2^56 + (h l' + l h') 2^28 + l l',
// and the last term (2^-62 r.m.s. of 1 for sums of 128 products) is dropped.  The sums of the
// first two are exact 64-bit integers: by Cauchy-Schwarz |sum hh| <= 2^62 |x||y| and |sum of both
// cross terms| <= 2^58 sqrt(2 n) (|x| + |y|) over n complex products, below 2^63 for
// vectors of norm 1 and n <= 128 (2^58 x 16 x 2).  Operands are scaled by powers of two so that those norms
// hold; the result carries an absolute error of about 2^-60 of the norms, where the FP64 chain of
// the same sum has a relative one of sqrt(2 n) 2^-54.8 (tests compare both).
#pragma once

#include <stdint.h>

namespace kubo {
namespace fx {

constexpr int BITS = 59;   // fractional bits of a full-scale operand
constexpr int LB = 28;     // bits of the low limb

__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

// round(x 2^s) for |x| 2^s < 2^60, from the bit pattern (round half up of the magnitude)
__device__ __forceinline__ long long from_double(double x, int s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & ((1ull << 52) - 1);
  if (ex) m |= 1ull << 52;
  else ex = 1;
  const int sh = ex - 1075 + s;   // x 2^s = m 2^sh
  const unsigned long long q =
      sh >= 0 ? m << (sh & 63) : (sh > -64 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
  return (long long)(b >> 63) ? -(long long)q : (long long)q;
}

// limbs of X
__device__ __forceinline__ int2 limbs(long long X) {
  return make_int2((int)((X + (1ll << (LB - 1))) >> LB), ((int)((uint32_t)X << (32 - LB))) >> (32 - LB));
}
__device__ __forceinline__ int4 climbs(long long re, long long im) {
  const int2 a = limbs(re), b = limbs(im);
  return make_int4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ long long value(int h, int l) { return ((long long)h << LB) + l; }

// running complex sum: products of the high limbs and the two cross products
struct Acc {
  long long rh, rm, ih, im;
};
__device__ __forceinline__ void zero(Acc& a) { a.rh = a.rm = a.ih = a.im = 0; }
__device__ __forceinline__ void mad(long long& acc, int a, int b) { acc += (long long)a * b; }

// acc += a b for complex limbs; (nyh, nyl) = -Im a
__device__ __forceinline__ void cmad(Acc& c, const int4& a, int nyh, int nyl, const int4& b) {
  mad(c.rh, a.x, b.x); mad(c.rm, a.x, b.y); mad(c.rm, a.y, b.x);
  mad(c.rh, nyh, b.z); mad(c.rm, nyh, b.w); mad(c.rm, nyl, b.z);
  mad(c.ih, a.x, b.z); mad(c.im, a.x, b.w); mad(c.im, a.y, b.z);
  mad(c.ih, a.z, b.x); mad(c.im, a.z, b.y); mad(c.im, a.w, b.x);
}
// acc += conj(a) b; (nyh, nyl) = -Im a
__device__ __forceinline__ void cmadc(Acc& c, const int4& a, int nyh, int nyl, const int4& b) {
  mad(c.rh, a.x, b.x); mad(c.rm, a.x, b.y); mad(c.rm, a.y, b.x);
  mad(c.rh, a.z, b.z); mad(c.rm, a.z, b.w); mad(c.rm, a.w, b.z);
  mad(c.ih, a.x, b.z); mad(c.im, a.x, b.w); mad(c.im, a.y, b.z);
  mad(c.ih, nyh, b.x); mad(c.im, nyh, b.y); mad(c.im, nyl, b.x);
}
// An operand that does not change in the loop that multiplies with it passes through pin() inside the
// loop: its widening to 64 bits would otherwise be moved out of the loop and every product become one of
// 64 by 64 bits, three multiply instructions (k_fixed.cu's reflectors: 309,000 -> 186,000 instructions of that
// pipe per k-point at W = 64).
__device__ __forceinline__ int4 pin(int4 v) {
  asm volatile("" : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w));
  return v;
}
// the sum at scale 2^(sx + sy - 56): hh + round(cross 2^-28)
__device__ __forceinline__ long long fold(long long h, long long m) {
  return h + ((m + (1ll << (LB - 1))) >> LB);
}
// round(v 2^-s), s >= 1, halves to the even neighbour: every 2^s-th v is a half, and always up they would add
// a constant to whatever the results are summed into
__device__ __forceinline__ long long rshift(long long v, int s) {
  return (v + (1ll << (s - 1)) - 1 + ((v >> s) & 1)) >> s;
}
// round((hh + cross 2^-28) 2^-s), s >= 1: rounded once.  (fold() and then a shift by one bit rounds every other value
// up from a half: a quarter unit too much on average in every entry of a rank-2 update, 46 units in
// the matrix norm at W = 128 where the roundings themselves are 9.)
__device__ __forceinline__ long long fold_shift(long long h, long long m, int s) {
  return (h + (m >> LB) + (1ll << (s - 1))) >> s;
}

// v 2^e (normal range) with the power of two added to the exponent field
__device__ __forceinline__ double to_double(long long v, int e) {
  const long long b = __double_as_longlong((double)v);
  return __longlong_as_double(v == 0 ? 0ll : b + ((long long)e << 52));
}
// x 2^e in FP64 for any e (the multiplier of an extreme exponent in two factors)
__device__ __forceinline__ double scale_pow2(double x, int e) {
  if (e >= -1000 && e <= 1000) return x * __longlong_as_double((long long)(1023 + e) << 52);
  return ldexp(x, e);
}

}  // namespace fx
}  // namespace kubo
