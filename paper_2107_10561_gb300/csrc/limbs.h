// Two-limb integers of FP64 values: what the INT32 pipe multiplies in place of the FP64 pipe.
// A value with |v| < 2^e is kept as the 58-bit integer v * 2^(58 - e) = h * 2^30 + l with a balanced low limb,
// |h| <= 2^28 and |l| <= 2^29. The product of two such values is h h' * 2^60 + (h l' + l h') * 2^30 + l l': three
// 32 x 32 -> 64 bit multiply-adds (4.3 clocks per warp and sub-core each, an FP64 multiply-add takes 64), and
// sums of them are exact. What is left out (l l') and what the limbs cut off lie about 2^-57 below the product of
// the two scales. FP64 loses 2^-53 of every term instead, so the scales have to follow the terms: every kernel here
// keeps a scale per class of unknowns (a velocity component or the pressure of one time node) on both sides and
// checks the sum of magnitudes it can see against the largest product of scales; a row that fails is summed in FP64.
#pragma once

#include <cstdint>

namespace stm {

constexpr int kLimbBits = 30, kLimbTotal = 58;

__device__ __forceinline__ int2 split_limbs(long long q) {
  return make_int2((int)((q + (1ll << (kLimbBits - 1))) >> kLimbBits), (int)((unsigned)q << (32 - kLimbBits)) >> (32 - kLimbBits));
}

// v * 2^(58 - e) rounded to an integer, |v| < 2^e
__device__ __forceinline__ long long fixed_of(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (ex) m |= 1ull << 52;
  const int sh = (ex ? ex : 1) - 1075 + kLimbTotal - e;  // <= 5 since |v| < 2^e
  if (sh >= 0) m <<= sh < 6 ? sh : 5;
  else if (sh > -55) m = (m + (1ull << (-sh - 1))) >> -sh;
  else m = 0;
  return (b >> 63) ? -(long long)m : (long long)m;
}
// the same as two limbs (x: high, y: low)
__device__ __forceinline__ int2 limbs_of(double v, int e) { return split_limbs(fixed_of(v, e)); }

// The same cut off instead of rounded, with a biased exponent: |v| < 2^(top - 1022), 64 <= top < 2047 (values of less
// than 2^-58 times that, zero and denormal ones among them, become zero)
__device__ __forceinline__ unsigned long long magnitude_below(double v, int top) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned s = (unsigned)(top + 6) - ((hi >> 20) & 0x7FFu);
  const unsigned a1 = __funnelshift_l(lo, hi, 11) | 0x80000000u, a0 = lo << 11;  // 53 bits at the top of 64
  unsigned long long q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(((unsigned long long)a1 << 32) | a0), "r"(s));  // 0 from 64 on
  return q;
}
__device__ __forceinline__ long long fixed_below(double v, int top) {
  const long long sg = __double2hiint(v) >> 31;
  return ((long long)magnitude_below(v, top) ^ sg) - sg;
}
// as two limbs that are not balanced (|h| < 2^28, |l| < 2^30)
__device__ __forceinline__ int2 limbs_below(double v, int top) {
  const unsigned long long q = magnitude_below(v, top);
  const int h = (int)(unsigned)(q >> kLimbBits), l = (int)((unsigned)q & ((1u << kLimbBits) - 1)), sg = __double2hiint(v) >> 31;
  return make_int2((h ^ sg) - sg, (l ^ sg) - sg);
}

// h, m += a * x: the sum is (h * 2^30 + m) * 2^30. As instructions of its own: where a limb comes out of a 64-bit
// shift the compiler multiplies 64-bit numbers, five times the instructions.
__device__ __forceinline__ void wide_fma(int a, int x, long long& c) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(x));
}
__device__ __forceinline__ void limb_fma(int2 a, int2 x, long long& h, long long& m) {
  wide_fma(a.x, x.x, h);
  wide_fma(a.x, x.y, m);
  wide_fma(a.y, x.x, m);
}

}  // namespace stm
