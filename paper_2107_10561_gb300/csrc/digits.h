// Balanced base-256 digits of FP64 values: what the tensor-core products of FP64 data are made of.
// FP64 arithmetic on this device issues 2 FMAs per clock and SM; FP16 tensor instructions with FP32
// accumulators run about 500 times as many multiplications, and products of 8-bit digits add up in them
// exactly as long as a sum stays below 2^24.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

namespace stm {

constexpr int kDig = 8;                     // digits of a 63-bit integer
constexpr int kExpZero = (int)0xA0A0A0A0;   // exponent of zero (a byte pattern): every digit is zero

// exponent e with |v| < 2^e (kExpZero for zero; 1025 for infinities and NaN)
__device__ __forceinline__ int exp_above(double v) {
  const int hi = __double2hiint(v) & 0x7FFFFFFF, lo = __double2loint(v);
  if ((hi | lo) == 0) return kExpZero;
  const int ex = hi >> 20;
  return ex == 0 ? -1021 : ex - 1022;
}

// v * 2^(62 - e) rounded to an integer, |v| < 2^e, as eight balanced digits (-128 .. 127) each biased by
// 128: byte 7 is digit 0, the most significant. Integer operations only.
__device__ __forceinline__ unsigned long long digits_of(double v, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (ex) m |= 1ull << 52;
  const int sh = (ex ? ex : 1) - 1075 + 62 - e;  // <= 9 since |v| < 2^e
  unsigned long long q;
  if (sh >= 0) q = m << (sh < 10 ? sh : 9);
  else if (sh > -55) q = (m + (1ull << (-sh - 1))) >> -sh;
  else q = 0;
  const long long sq = (b >> 63) ? -(long long)q : (long long)q;
  return (unsigned long long)sq + 0x8080808080808080ull;
}
// digit d (0 = most significant) as FP16: 1024 + byte is 0x6400 | byte
__device__ __forceinline__ __half digit_half(unsigned long long p, int d) {
  const unsigned short h = (unsigned short)(0x6400u | (unsigned)((p >> (56 - 8 * d)) & 0xFFu));
  return __hsub(__ushort_as_half(h), __ushort_as_half(0x6480));
}

// Two neighbouring values as one register set: words i: bytes u_i, u_{i+4}, v_i, v_{i+4} of two packs (digit i is byte 7 - i of a pack)
__device__ __forceinline__ uint4 words_of(unsigned long long u, unsigned long long v) {
  const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u, vh = (uint32_t)(v >> 32), vl = (uint32_t)v;
  const uint32_t a = __byte_perm(uh, ul, 0x6273), b = __byte_perm(uh, ul, 0x4051);  // u0 u4 u1 u5 | u2 u6 u3 u7
  const uint32_t c = __byte_perm(vh, vl, 0x6273), d = __byte_perm(vh, vl, 0x4051);
  return make_uint4(__byte_perm(a, c, 0x5410), __byte_perm(a, c, 0x7632), __byte_perm(b, d, 0x5410),
                    __byte_perm(b, d, 0x7632));
}
// digit s of the two positions of a word, as a pair of FP16 integers
__device__ __forceinline__ uint32_t digit_pair(uint32_t w, bool low) {
  const uint32_t h = __byte_perm(w, 0x64646464u, low ? 0x4341 : 0x4240), bias = 0x64806480u;
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), *reinterpret_cast<const __half2*>(&bias));
  return *reinterpret_cast<const uint32_t*>(&d);
}

__device__ __forceinline__ void mma_f16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// v * 2^e without intermediate overflow or underflow
__device__ __forceinline__ double scale_pow2(double v, int e) {
  if (e > -900 && e < 900) return v * __hiloint2double((e + 1023) << 20, 0);
  return ldexp(v, e);
}

// Sums of fewer than 2^22 in magnitude may start from kSumZero: 1.5 x 2^23, so that the sum's integer stands in
// the low bits of the FP32 pattern (a conversion would run at an eighth of the FMA rate).
constexpr float kSumZero = 12582912.f;
// hi (digits 0 .. 3) and lo (4 .. 7) of eight such sums: sum_d s_d 256^(3 - d)
__device__ __forceinline__ void join_sums(const float (*acc)[4], int m, long long& hi, long long& lo) {
  constexpr long long zero = 0x4B400000ll * (16777216 + 65536 + 256 + 1);
  hi = lo = -zero;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    hi += (long long)__float_as_int(acc[d][m]) * (1 << (24 - 8 * d));
    lo += (long long)__float_as_int(acc[d + 4][m]) * (1 << (24 - 8 * d));
  }
}
// (hi * 2^32 + lo) * 2^e, rounded once, with integer operations only: conversions and products would wait for
// the FP64 pipe. |hi| < 2^62.
__device__ __forceinline__ double join_pow2(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 32);
  uint32_t l = (uint32_t)lo;  // the value is h * 2^32 + l
  const bool neg = h < 0;
  if (neg) {
    h = l ? ~h : -h;
    l = 0u - l;
  }
  unsigned long long u = (unsigned long long)h;
  if (u == 0) {
    if (l == 0) return 0.0;
    u = l;
    l = 0;
    e -= 32;
  }
  const int lz = __clzll((long long)u), ex = 1023 + 63 + 32 - lz + e;
  u = (u << lz) | (((unsigned long long)l << 32) >> (64 - lz));  // lz >= 1
  if (ex < 1 || ex > 2045) {
    const double v = scale_pow2((double)u, 32 - lz + e);
    return neg ? -v : v;
  }
  u = (u >> 11) + ((u >> 10) & 1);  // 53 bits, the rounding may carry into the exponent
  u += ((unsigned long long)(ex - 1) << 52);
  return __longlong_as_double((long long)(u | (neg ? 0x8000000000000000ull : 0ull)));
}
// |v| as an integer key that orders like |v|; NaN orders below everything
__device__ __forceinline__ long long abs_key(double v) {
  const long long k = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll;
  return k > 0x7FF0000000000000ll ? -1 : k;
}

}  // namespace stm
