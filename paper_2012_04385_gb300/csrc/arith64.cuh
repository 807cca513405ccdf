// IEEE FP64 division and square root, correctly rounded, on the integer pipe.
//
// On GB300 the FP64 pipe issues one warp instruction per 16 cycles and SM (two
// lanes per cycle), 1/64 of the FP32 and integer rate, and a double division or
// square root is a chain of about ten FP64 instructions there.  The FP64 stage
// needs some 70 divisions per face, which made them the larger half of its
// FP64-pipe time.  Here the quotient's 54 leading bits are found by schoolbook
// long division in two digits of about 2^30 and 2^24 (Knuth, TAOCP vol. 2,
// sec. 4.3.1: a quotient digit estimated from the leading parts, then corrected
// by the exact remainder), the estimates from an FP32 reciprocal of the
// divisor's leading 24 bits sharpened once in 32-bit integers; the square root
// is found in the same two digits (digit-by-digit root with exact remainder).
// The remainders are exact integers, so the results do not depend on the
// accuracy of the FP32 seed beyond the stated bounds.
//
// A quotient (or root) of 53-bit operands never lies half way between two
// 53-bit numbers, so the 54-bit truncation decides the rounding.
//
// Operands outside the normal range, quotients near its ends and NaN take the
// compiler's operation; a zero numerator is answered directly (x / rho at rest
// is the common case, and there the compiler's division leaves its fast path).
//
// A division is some 45 integer instructions, less than the issue time of one
// FP64 instruction (64 slots); figures of the stage at k_flux_f64 (rhs.cuh).
#pragma once

#include <cstdint>
#include <cstring>

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mrb {

__host__ __device__ __forceinline__ uint64_t d2bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double bits2d(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float seed_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float seed_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#else
extern float seed_rcp(float x);      // host checks: any value within 2^-21 of 1/x, or of 1/sqrt(x)
extern float seed_rsqrt(float x);
#endif

__host__ __device__ __forceinline__ uint32_t f2bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float bits2f(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

// The divisor's part of a division, shared by all quotients of one divisor.
struct Div64 {
  double b;
  uint64_t m;        // mantissa with the leading bit, in [2^52, 2^53)
  uint32_t x;        // X = 2^83 / m within 3
  int32_t e;         // biased exponent; 0 or 2047 for operands left to the compiler's division
};

__host__ __device__ __forceinline__ Div64 div64_prep(double b) {
  Div64 d;
  const uint64_t w = d2bits(b);
  const uint32_t hi = (uint32_t)(w >> 32);
  d.b = b;
  d.e = (int32_t)((hi >> 20) & 2047u);
  d.m = (w & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const uint32_t bh = (uint32_t)(d.m >> 21);                       // leading 32 bits, in [2^31, 2^32)
  // r = 1/b of the leading 24 bits within 2^-22, kept in [1/2, 1)
  const float r = seed_rcp(bits2f(0x3F800000u | ((bh >> 8) & 0x007FFFFFu)));
  uint32_t rb = f2bits(r);
  rb = rb > 0x3F7FFFFFu ? 0x3F7FFFFFu : (rb < 0x3F000000u ? 0x3F000000u : rb);
  const uint32_t x0 = ((rb & 0x007FFFFFu) | 0x00800000u) << 7;      // r 2^31, below 2^31
  // one Newton step: x0 (2 - b x0), b x0 = bh x0 / 2^62
  const int32_t t = (int32_t)(((uint64_t)bh * x0) >> 30);          // (b x0) 2^32 modulo 2^32: the defect, negated
  d.x = x0 - (uint32_t)(((int64_t)t * (int64_t)(int32_t)x0) >> 32);
  return d;
}

__host__ __device__ __forceinline__ double div64(double a, const Div64& d) {
  const uint64_t w = d2bits(a), s = (w ^ d2bits(d.b)) & 0x8000000000000000ull;
  const int32_t ea = (int32_t)((uint32_t)(w >> 52) & 2047u);
  const int32_t e = ea - d.e + 1022;                               // exponent of the quotient, or one less
  const bool ok = (uint32_t)(ea - 1) < 2046u && (uint32_t)(d.e - 1) < 2046u && (uint32_t)(e - 1) < 2044u;
  if (!ok) {
    // a zero over a normal number is a zero of the right sign
    if ((w << 1) == 0 && (uint32_t)(d.e - 1) < 2046u) return bits2d(s);
    return a / d.b;
  }
  const uint64_t ma = (w & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  // first digit: ma 2^30 / m, less 1 .. 8.5 (the estimate is off by -3 .. 4.5: 3 from
  // x, 1/2 and 1 from the two truncations; 4 is taken off)
  const uint32_t q1 = mulhi32((uint32_t)(ma >> 21), d.x) - 4u;
  const uint64_t r1 = (ma << 30) - (uint64_t)q1 * d.m;             // exact: m < r1 < 9 m < 2^57
  // second digit: r1 2^24 / m < 9 2^24, less 0.5 .. 2.6 (off by -0.5 .. 1.6, 1 taken off)
  const uint32_t q2 = (mulhi32((uint32_t)(r1 >> 25), d.x) >> 2) - 1u;
  uint64_t r2 = (r1 << 24) - (uint64_t)q2 * d.m;                   // modulo 2^64; the true value is below 3 m
  uint64_t q = ((uint64_t)q1 << 24) + q2;                          // floor(ma 2^54 / m) less 0 .. 2
  if (r2 >= d.m) { r2 -= d.m; ++q; }
  if (r2 >= d.m) ++q;
  // q in (2^53, 2^55): keep 54 bits, round on the last
  const uint32_t big = (uint32_t)(q >> 54);                        // 1 when ma >= m
  const uint64_t m = ((q >> big) + 1u) >> 1;                       // [2^52, 2^53]
  return bits2d(s | (((uint64_t)(uint32_t)(e + (int32_t)big - 1) << 52) + m));
}

__host__ __device__ __forceinline__ double div64(double a, double b) { return div64(a, div64_prep(b)); }

// The divisor part of a small integer (at compile time).
__host__ __device__ constexpr Div64 div64_of(uint32_t n) {
  int lg = 0;
  while ((n >> (lg + 1)) != 0) ++lg;
  return Div64{(double)n, (uint64_t)n << (52 - lg), (uint32_t)((1ull << (31 + lg)) / n), 1023 + lg};
}

// x / 6: the 56-bit numerator 8 ma over 3 in two digits of 28 bits.
__host__ __device__ __forceinline__ double div64_6(double a) {
  const uint64_t w = d2bits(a), s = w & 0x8000000000000000ull;
  const int32_t ea = (int32_t)((uint32_t)(w >> 52) & 2047u);
  if ((uint32_t)(ea - 4) >= 2043u) return (w << 1) == 0 ? a : a / 6.0;
  const uint64_t ma = (w & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const uint64_t n = ma << 3;
  const uint32_t nh = (uint32_t)(n >> 28), qh = mulhi32(nh, 0xAAAAAAABu) >> 1;
  const uint32_t nl = ((nh - 3u * qh) << 28) | ((uint32_t)n & 0x0FFFFFFFu), ql = mulhi32(nl, 0xAAAAAAABu) >> 1;
  const uint64_t q = ((uint64_t)qh << 28) + ql;                    // floor(8 ma / 3) in (2^53, 2^55)
  const uint32_t big = (uint32_t)(q >> 54);
  const uint64_t m = ((q >> big) + 1u) >> 1;
  return bits2d(s | (((uint64_t)(uint32_t)(ea - 4 + (int32_t)big) << 52) + m));
}

// sqrt(x), correctly rounded: the 54-bit root of M 2^54 (M the mantissa, one bit
// longer for odd exponents) as s1 2^26 + s2 with s1 = floor(sqrt(4 M)).
__host__ __device__ __forceinline__ double sqrt64(double x) {
  const uint64_t w = d2bits(x);
  const int32_t ex = (int32_t)(uint32_t)(w >> 52);                  // sign bit included
  if ((uint32_t)(ex - 1) >= 2046u) {
#ifdef __CUDA_ARCH__
    return sqrt(x);
#else
    return std::sqrt(x);
#endif
  }
  const uint32_t odd = (uint32_t)(ex + 1) & 1u;                     // exponent ex - 1023 odd
  const uint64_t M = ((w & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << odd;   // v = M / 2^52 in [1, 4)
  const uint32_t Mh = (uint32_t)(M >> 22);                         // v 2^30
  // y = 1/sqrt(v) in (1/2, 1] within 2^-21, as y 2^31 below 2^31
  const float f = bits2f((odd ? 0x40000000u : 0x3F800000u) | ((uint32_t)(w >> 29) & 0x007FFFFFu));
  const float r = seed_rsqrt(f);
  uint32_t rb = f2bits(r);
  rb = rb > 0x3F7FFFFFu ? 0x3F7FFFFFu : (rb < 0x3F000000u ? 0x3F000000u : rb);
  const uint32_t y0 = ((rb & 0x007FFFFFu) | 0x00800000u) << 7;
  // one Newton step, y += y (1 - v y^2) / 2
  const uint32_t vy = mulhi32(Mh, y0);                             // v y 2^29
  const int32_t t = (int32_t)(((uint64_t)vy * y0) >> 28);          // v y^2 2^32 modulo 2^32: the defect, negated
  const uint32_t y = y0 - (uint32_t)(((int64_t)t * (int64_t)(int32_t)y0) >> 33);
  // s1 = floor(sqrt(4 M)), the estimate v y 2^27 off by less than 2 and corrected
  uint32_t s1 = (mulhi32(Mh, y) >> 2);
  int64_t r1 = (int64_t)((M << 2) - (uint64_t)s1 * s1);
  if (r1 < 0) { --s1; r1 += 2 * (int64_t)s1 + 1; }
  if (r1 < 0) { --s1; r1 += 2 * (int64_t)s1 + 1; }
  if (r1 > 2 * (int64_t)s1) { r1 -= 2 * (int64_t)s1 + 1; ++s1; }
  if (r1 > 2 * (int64_t)s1) { r1 -= 2 * (int64_t)s1 + 1; ++s1; }
  // s2 = floor of the rest, estimated as r1 2^25 / s1 = r1 y / 2^33
  uint32_t s2 = (uint32_t)(((uint64_t)(uint32_t)r1 * y) >> 33);
  const uint64_t s = ((uint64_t)s1 << 26) + s2;
  const int64_t r2 = (int64_t)(((((uint64_t)r1 << 25) - (uint64_t)s1 * s2) << 27) - (uint64_t)s2 * s2);
  const uint64_t sc = s + (r2 > 2 * (int64_t)s ? 1u : 0u) - (r2 < 0 ? 1u : 0u);
  const uint64_t m = (sc + 1u) >> 1;
  return bits2d(((uint64_t)(uint32_t)(((ex - 1023 - (int32_t)odd) >> 1) + 1022) << 52) + m);
}

// The mean 0.125 (((u0 + u1) + (u2 + u3)) + ((u4 + u5) + (u6 + u7))), each sum
// rounded to nearest even.  Values of one sign and exponent (the usual eight
// children of a cell): a sum of two has the next exponent and drops one bit, so
// each level of sums is a rounded mean of 52-bit fractions; about 65 integer
// instructions for eight of the FP64 pipe, which cost 64 issue slots each.  The
// last sum's exponent is three above, so it stays finite.  Eight equal values
// without an exponent (zeros) are their own mean.
__host__ __device__ __forceinline__ uint64_t mean_even(uint64_t a, uint64_t b) {
  const uint64_t x = a + b, q = x >> 1;
  return q + (x & q & 1u);
}
__host__ __device__ __forceinline__ double mean8(const double (&v)[8]) {
  constexpr uint64_t M = 0x000fffffffffffffull;
  const uint64_t u0 = d2bits(v[0]);
  uint64_t d = 0;
#pragma unroll
  for (int i = 1; i < 8; ++i) d |= d2bits(v[i]) ^ u0;
  const uint32_t e = (uint32_t)(u0 >> 52) & 2047u;
  if (e == 0 ? d == 0 : (d <= M && e < 2043u)) {
    if (e == 0) return v[0];
    uint64_t m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = mean_even(d2bits(v[2 * i]) & M, d2bits(v[2 * i + 1]) & M);
    return bits2d((u0 & ~M) | mean_even(mean_even(m[0], m[1]), mean_even(m[2], m[3])));
  }
  return 0.125 * (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])));
}

}  // namespace mrb
