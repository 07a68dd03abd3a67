// c2f_exact.cuh -- binary64 division, square root and rounding to integers on
// the integer units.
//
// A GB300 SM retires two FP64 operations a clock against 64 or more 32-bit
// integer ones, so an FP64 instruction costs a warp 16 cycles of the SM's only
// FP64 pipe and a correctly rounded division or square root, some eight or nine
// of them in a row, about 140.  The functions below return the same correctly
// rounded results (IEEE-754, to nearest even: the result is unique, however it
// is computed) from 32 x 32 -> 64-bit integer products, in about 60
// instructions that run beside the FP64 pipe.  Division: a 32-bit reciprocal
// estimate, one Newton step in integers, the 53-bit quotient and its exact
// remainder.  Square root: a 32-bit reciprocal root, one Newton step, a 32-bit
// root with its exact remainder, and the remaining 21 bits by one linear step
// from that remainder, then the exact remainder of all 53.  The remainder
// decides the rounding.  Arguments outside the stated ranges (zeros,
// subnormals, infinities, NaN, extreme exponents) take the FP64 instructions.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define C2F_HD __host__ __device__ __forceinline__
#else
#define C2F_HD inline
#include <cmath>
#endif

namespace c2f {

C2F_HD uint64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
C2F_HD double double_of(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}
C2F_HD uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
C2F_HD uint32_t mul_hi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// estimates of 1/x and 1/sqrt(x), good to about 2^-22 relative (host builds may
// scale theirs, to stand for the error of the GPU's)
#ifndef C2F_HOST_ESTIMATE_SCALE
#define C2F_HOST_ESTIMATE_SCALE 1.0f
#endif
C2F_HD float rcp_estimate(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return (1.0f / x) * (C2F_HOST_ESTIMATE_SCALE);
#endif
}
C2F_HD float rsqrt_estimate(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return (1.0f / sqrtf(x)) * (C2F_HOST_ESTIMATE_SCALE);
#endif
}
// truncation to uint32, larger values to 2^32 - 1
C2F_HD uint32_t to_u32(float x) {
#ifdef __CUDA_ARCH__
  return __float2uint_rz(x);
#else
  return x >= 4294967296.0f ? 0xFFFFFFFFu : (uint32_t)x;
#endif
}

// positive, 2^-500 <= x < 2^500 (from the high word)
C2F_HD bool mid_range(uint64_t bits) { return (uint32_t)(bits >> 32) - (523u << 20) < (1000u << 20); }

// RN(x / y) for x and y both positive in mid_range
C2F_HD double div_mid(double x, double y) {
  const uint64_t bx = bits_of(x), by = bits_of(y);
  const uint64_t m52 = 0x000FFFFFFFFFFFFFull, one = 0x0010000000000000ull;
  const uint64_t ma = (bx & m52) | one, mb = (by & m52) | one;   // significands, 53 bits
  const uint32_t b1 = (uint32_t)(mb >> 21), b0 = (uint32_t)(mb << 11);   // B = mb 2^11, [2^63, 2^64)
  const uint32_t a1 = (uint32_t)(ma >> 21), a0 = (uint32_t)(ma << 11);
  // r0 ~ 2^95 / B, relative error d0 <= 2^-22; a Newton step r = r0 2^32 (1 + (1 - r0 B / 2^95)):
  // 2^127 / B less its relative error d0^2 <= 2^-44
  const uint32_t r0 = to_u32(rcp_estimate((float)b1) * 0x1p63f);
  const uint64_t p = wide(b1, r0) + mul_hi(b0, r0);               // r0 B / 2^32 ~ 2^63
  const int32_t d = (int32_t)((int64_t)(0x8000000000000000ull - p) >> 11);
  const uint64_t r = ((uint64_t)r0 << 32) + (uint64_t)(((int64_t)d * (int32_t)(r0 >> 1)) >> 19);
  const uint32_t r1 = (uint32_t)(r >> 32), rl = (uint32_t)r;
  // h ~ (ma / mb) 2^63, less than the exact value (the product's low parts are
  // dropped and 8 is taken off); q: its first 53 bits, short of the quotient by
  // at most 2^10
  const uint64_t h = wide(a1, r1) + mul_hi(a1, rl) + mul_hi(a0, r1) - 8u;
  const int less = ma < mb ? 1 : 0;
  uint64_t q = h >> (11 - less);
  const uint64_t rem = (ma << (52 + less)) - q * mb;              // exact modulo 2^64, < 2^63
  // the rest of the quotient, short by at most 1
  const uint32_t dq = mul_hi((uint32_t)(rem >> 31), r0 - 2048u) >> 21;
  uint64_t left = rem - (uint64_t)dq * mb;
  const bool up = left >= mb;
  left -= up ? mb : 0ull;
  // round to nearest by the remainder (a quotient of 53-bit numbers is never a tie)
  q += dq + (up ? 1u : 0u) + (2 * left > mb ? 1u : 0u);
  const uint32_t e = (uint32_t)(bx >> 52) - (uint32_t)(by >> 52) + 1022u - (uint32_t)less;
  return double_of(q + ((uint64_t)e << 52));
}

// RN(sqrt(x)) for x positive in mid_range
C2F_HD double sqrt_mid(double x) {
  const uint64_t bx = bits_of(x);
  const uint32_t e = (uint32_t)(bx >> 52);
  // x = N 2^(2 k), N in [2^62, 2^64): the root of N 2^42 has 53 bits
  const uint64_t n = ((bx & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << (10 + ((e & 1u) ^ 1u));
  const uint32_t n1 = (uint32_t)(n >> 32);
  // y ~ 2^63 / sqrt(N) (32 bits, [2^31, 2^32]); a Newton step brings 2^-22 to about 2^-31
  uint32_t y = to_u32(rsqrt_estimate((float)n1) * 0x1p47f);
  const uint32_t y2 = mul_hi(y, y);                              // y^2 / 2^32
  const int32_t d = (int32_t)(0x40000000u - mul_hi(n1, y2));     // 2^30 (1 - N y^2 / 2^126)
  const int64_t yn = (int64_t)y + (((int64_t)d * (int32_t)(y >> 1)) >> 30);
  y = yn > 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)yn;
  // s ~ sqrt(N), 32 bits, and what it leaves of N; s is off by a few units
  const uint64_t s64 = (wide(n1, y) + mul_hi((uint32_t)n, y)) >> 31;
  const uint32_t s = s64 >> 32 ? 0xFFFFFFFFu : (uint32_t)s64;
  const int64_t rem = (int64_t)(n - wide(s, s));                 // |rem| < 2^37
  // + rem / (2 s) = rem y / 2^64, to 21 bits more
  int64_t q = ((int64_t)s << 21) + ((((rem >> 6) * (int64_t)(y >> 1)) >> 36));
  int64_t left = (int64_t)((n << 42) - (uint64_t)q * (uint64_t)q);   // exact: q is off by a few units
  if (left < 0) { --q; left += 2 * q + 1; }
  if (left > 2 * q) { left -= 2 * q + 1; ++q; }
  // now q = floor(root): up when the root lies past q + 1/2 (never on it)
  q += left > q ? 1 : 0;
  return double_of((uint64_t)q + ((uint64_t)((e + 1021u) >> 1) << 52));
}

// RN(x y) for x and y both positive in mid_range: the 128-bit product of the
// significands, its dropped bits gathered in the last one kept
C2F_HD double mul_mid(double x, double y) {
  const uint64_t bx = bits_of(x), by = bits_of(y);
  const uint32_t a1 = (uint32_t)(bx >> 21) | 0x80000000u, a0 = (uint32_t)(bx << 11);
  const uint32_t b1 = (uint32_t)(by >> 21) | 0x80000000u, b0 = (uint32_t)(by << 11);
  const uint64_t w0 = wide(a0, b0);
  const uint64_t w1 = wide(a1, b0) + (w0 >> 32);
  const uint64_t w2 = wide(a0, b1) + (uint32_t)w1;
  uint64_t h = wide(a1, b1) + (w1 >> 32) + (w2 >> 32);            // [2^62, 2^64)
  const uint32_t top = (uint32_t)(h >> 63);
  h = (h << (1u - top)) | (((uint32_t)w0 | (uint32_t)w2) != 0u ? 1u : 0u);
  uint64_t q = h >> 11;
  q += ((uint32_t)h & 0x7FFu) + ((uint32_t)q & 1u) > 0x400u ? 1u : 0u;   // to nearest, ties to even
  const uint32_t e = (uint32_t)(bx >> 52) + (uint32_t)(by >> 52) - 1024u + top;
  return double_of(q + ((uint64_t)e << 52));
}

// 2^-500 <= x < 1
C2F_HD bool below_one(uint64_t bits) { return (uint32_t)(bits >> 32) - (523u << 20) < (500u << 20); }

// RN(1 - x) for x in below_one: in units of 2^-53 it is 2^53 less x rounded to
// an integer when x < 1/2, and exact when x >= 1/2
C2F_HD double one_minus(double x) {
  const uint64_t b = bits_of(x);
  const uint64_t m = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  uint32_t s = 1022u - (uint32_t)(b >> 52);                       // x = m 2^-(53 + s)
  s = s > 60u ? 60u : s;                                          // far below 1/2: no integer part, no half
  const uint64_t k = m >> s, rest = (m << 3) << (61u - s);         // rest: the fraction, as 64 bits
  const bool up = rest > 0x8000000000000000ull || (rest == 0x8000000000000000ull && (k & 1u));
  const uint64_t n = 0x20000000000000ull - k - (up ? 1u : 0u);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)n);
#else
  const int lz = __builtin_clzll(n);
#endif
  const uint32_t left = lz > 11 ? (uint32_t)lz - 11u : 0u;
  return double_of((n << left) + ((uint64_t)(1021u - left) << 52));
}

// ---- the Horner steps of exp and log
// q = c + p r for a p of 53 bits and |r| < 2^-7, each sum rounded to binary64:
// the exponents of every c and q are known ahead, so with r as a 64-bit integer
// A 2^-70 (exact for |r| >= 2^-18) a step is the high part of one product, at
// 17 to 19 bits below the sum's last place, rounded and added to c's
// significand.  The dropped parts are under 3 units of the product's last
// place, so a step is exact unless those bits lie within 3 of a half; then (one
// argument in 20,000), and for smaller r, `exact` stays false and the caller
// takes the FP64 instructions.
struct HornerArg {
  uint32_t a1, a0;
  bool exact;
  C2F_HD explicit HornerArg(double r) {
    const uint64_t b = bits_of(r);
    const uint32_t e = (uint32_t)(b >> 52) & 0x7FFu;
    exact = e - 1005u <= 10u;
    const uint64_t a = ((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << ((e - 1005u) & 15u);
    a1 = (uint32_t)(a >> 32);
    a0 = (uint32_t)a;
  }
  // round(n A 2^-(53 + guard)) for a 53-bit n
  C2F_HD uint64_t times(uint64_t n, int guard) {
    const uint32_t n1 = (uint32_t)(n >> 21), n0 = (uint32_t)(n << 11), half = 1u << (guard - 1);
    const uint64_t x = wide(n1, a1) + mul_hi(n1, a0) + mul_hi(n0, a1) + half;
    exact = exact && (((uint32_t)x + 3u) & (2u * half - 1u)) > 3u;
    return x >> guard;
  }
};

// significands of the constants, and the bits of 1/2
constexpr uint64_t kM1_120 = 0x11111111111111ull, kM1_24 = 0x15555555555555ull;   // 2^-59, 2^-57
constexpr uint64_t kM1_6 = 0x15555555555555ull, kM1_5 = 0x1999999999999Aull;      // 2^-55, 2^-55
constexpr uint64_t kM1_3 = 0x15555555555555ull, kBitsHalf = 0x3FE0000000000000ull;   // 2^-54

// ((1/120 r + 1/24) r + 1/6) r + 1/2
C2F_HD double exp_steps(double r, bool *exact) {
  HornerArg A(r);
  const bool neg = (bits_of(r) >> 63) != 0;
  const uint64_t x1 = A.times(kM1_120, 19), n1 = neg ? kM1_24 - x1 : kM1_24 + x1;
  const uint64_t x2 = A.times(n1, 19), n2 = neg ? kM1_6 - x2 : kM1_6 + x2;
  const uint64_t x3 = A.times(n2, neg ? 18 : 19);   // below 1/2 the last place is half as large
  *exact = A.exact;
  return double_of(neg ? kBitsHalf - x3 : kBitsHalf + x3);
}

// (((-1/6 r + 1/5) r - 1/4) r + 1/3) r - 1/2, for r > 0
C2F_HD double log_steps(double r, bool *exact) {
  HornerArg A(r);
  const uint64_t n1 = kM1_5 - A.times(kM1_6, 17);
  const uint64_t n2 = 0x20000000000000ull - A.times(n1, 17);   // 1/4 = 2^53 2^-55
  const uint64_t n3 = kM1_3 - A.times(n2, 18);
  const uint64_t x4 = A.times(n3, 17);
  *exact = A.exact && (bits_of(r) >> 63) == 0;
  return double_of(0x8000000000000000ull | (kBitsHalf - x4));
}

}  // namespace c2f
