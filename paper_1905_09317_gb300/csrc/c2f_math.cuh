// c2f_math.cuh -- device elementary functions, Philox4x32-10 and the ROS
// perturbation draw.
//
// Every exp / log / sin / cos on the fire-growth path is computed here from
// IEEE-754 primitives (correctly rounded +, *, /, sqrt and fused multiply-add,
// with no compiler contraction: the library is built with --fmad=false and
// the fused steps are explicit __fma_rn calls), so that a CPU build of the
// same construction reproduces every bit.  Constructions:
//   series forms (dexp_series, dlog_series), which fill the tables below:
//     exp   x = k ln2 + r (Cody-Waite, 29-bit head of ln2), Taylor to r^13, 2^k
//     log   x = 2^e m, m in [sqrt(1/2), sqrt(2)], 2 atanh((m-1)/(m+1)) to s^21
//   table forms (Tang's method), used everywhere else:
//     exp   x = (64k + j) ln2/64 + r: 2^k T_j (1 + p(r)), T_j = 2^(j/64),
//           p = Taylor of exp(r) - 1 to r^5
//     log   x = 2^e m, m in [1, 2), j = top 8 fraction bits, V_j = 1/(1 + j/256)
//           rounded, r = m V_j - 1 (one fused rounding):
//           e ln2 - log V_j + (Taylor of log(1 + r) to r^6)
//   sin/cos of degrees: exact reduction by multiples of 90, Taylor to t^17/t^18
//   pow(x, y) = x^n sqrt(x)^(2y odd) for y a positive multiple of 1/2 up to
//               8 (n = floor y, products from the left), else exp(y log x)
// and the same in binary32 (exp to r^7, log to s^11, cos of a fraction of a
// turn) for the perturbation draw.  Taylor coefficients are 1/k! as correctly
// rounded binary64 quotients; they live in __constant__ memory, filled once per
// device by upload_constants().
#pragma once
#include <cmath>
#include <cstdint>

#include "c2f_exact.cuh"
#include "c2f_layout.cuh"

namespace c2f {

// coefficient tables, filled once per device by upload_constants()
__constant__ MathConstants g_mc;
// exp / log tables (lanes index them independently, so global memory through
// the read-only cache rather than __constant__), filled by k_math_tables
__device__ double g_exp_tab[64];    // 2^(j/64)
__device__ double g_log_inv[256];   // RN(1 / (1 + j/256))
__device__ double g_log_tab[256];   // -log(g_log_inv[j])

// host: compute the coefficient tables (plain IEEE binary64 arithmetic)
inline void make_math_constants(MathConstants *m) {
  double f = 1.0;
  for (int k = 0; k < 24; ++k) {
    if (k > 0) f = f * (double)k;
    m->inv_fact[k] = 1.0 / f;
  }
  for (int n = 0; n < 12; ++n) m->log_c[n] = 1.0 / (double)(2 * n + 1);
  for (int n = 0; n < 10; ++n) {
    const double sgn = (n & 1) ? -1.0 : 1.0;
    m->sin_c[n] = sgn * m->inv_fact[2 * n + 1];
    m->cos_c[n] = sgn * m->inv_fact[2 * n];
  }
  for (int k = 0; k < 12; ++k) m->inv_fact_f[k] = (float)m->inv_fact[k];
  for (int n = 0; n < 8; ++n) m->log_cf[n] = (float)m->log_c[n];
  for (int n = 0; n < 8; ++n) {
    m->sin_cf[n] = (float)m->sin_c[n];
    m->cos_cf[n] = (float)m->cos_c[n];
  }
}

constexpr double kLn2Hi = 0x1.62e42ffp-1;            // 29 significant bits
constexpr double kLn2Lo = -0x1.718432a1b0e26p-35;    // ln2 - kLn2Hi, rounded
constexpr double kInvLn2 = 0x1.71547652b82fep+0;
constexpr double kDeg2Rad = 0x1.1df46a2529d39p-6;
constexpr double kSqrt2 = 0x1.6a09e667f3bcdp+0;
constexpr float kLn2HiF = 0x1.62ep-1f;               // 13 significant bits
constexpr float kLn2LoF = 0x1.0bfbe8p-15f;
constexpr float kInvLn2F = 0x1.715476p+0f;
constexpr float kTwoPiF = 0x1.921fb6p+2f;
constexpr float kSqrt2F = 0x1.6a09e6p+0f;

// Comparisons of a double with 0 or a positive constant as integer compares of
// the bit patterns (the order of non-NaN doubles against a positive constant is
// the order of their bits read as signed 64-bit integers).  The values tested
// on the rate-of-spread path are never NaN; these keep the compares off the
// FP64 unit, which the table kernel saturates.
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ bool pos(double x) { return dbits(x) > 0; }   // x > 0
__device__ __forceinline__ bool gt_c(double x, double c) { return dbits(x) > dbits(c); }   // x > c > 0
__device__ __forceinline__ bool lt_c(double x, double c) { return dbits(x) < dbits(c); }   // x < c, c > 0
__device__ __forceinline__ bool le_c(double x, double c) { return dbits(x) <= dbits(c); }  // x <= c, c > 0

__device__ __forceinline__ double pow2i(int k) {  // exact 2^k for -1022 <= k <= 1023
  return __longlong_as_double((long long)(k + 1023) << 52);
}

__device__ __forceinline__ double scale2(double p, int k) {
  if (k > 1023) return __dmul_rn(__dmul_rn(p, pow2i(1023)), pow2i(k - 1023));
  if (k < -1022) return __dmul_rn(__dmul_rn(p, pow2i(k + 600)), pow2i(-600));
  return __dmul_rn(p, pow2i(k));
}

// The rare FP64 steps of the routines below, out of line: inlined, the compiler
// predicates them instead of branching, and a predicated-off FP64 instruction
// takes its slot of the pipe all the same (the table kernel went from 180 only
// to 175 FP64 instructions a cell-hour when its exp and log steps moved to
// integers with the FP64 steps kept inline behind a test).
__device__ __noinline__ double ddiv_any(double x, double y) { return __ddiv_rn(x, y); }
__device__ __noinline__ double dsqrt_any(double x) { return __dsqrt_rn(x); }
__device__ __noinline__ double dmul_any(double x, double y) { return __dmul_rn(x, y); }
__device__ __noinline__ double dscale_any(double p, int k) { return scale2(p, k); }
__device__ __noinline__ double drint_product(double x, double y) { return rint(__dmul_rn(x, y)); }
__device__ __noinline__ double exp_steps_any(double r) {
  return __fma_rn(__fma_rn(__fma_rn(g_mc.inv_fact[5], r, g_mc.inv_fact[4]), r, g_mc.inv_fact[3]), r, g_mc.inv_fact[2]);
}
__device__ __noinline__ double log_steps_any(double r) {
  double q = __fma_rn(-g_mc.inv_fact[3], r, g_mc.log_c[2]);   // -1/6, 1/5
  q = __fma_rn(q, r, -0.25);
  q = __fma_rn(q, r, g_mc.log_c[1]);                          // 1/3
  return __fma_rn(q, r, -0.5);
}
__device__ __noinline__ double dexp_far(double x) {   // |x| >= 704 and not in (704, 709.78]: the value, else 1
  if (x != x) return x;
  if (x > 709.78) return __longlong_as_double(0x7ff0000000000000LL);
  return x < -745.2 ? 0.0 : 1.0;
}

// x / y and sqrt(x), correctly rounded: on the integer units over the range
// that the rates take, by the FP64 instructions elsewhere
__device__ __forceinline__ double ddiv(double x, double y) {
  return mid_range(bits_of(x)) && mid_range(bits_of(y)) ? div_mid(x, y) : ddiv_any(x, y);
}
// x y for x, y >= 0 and 1 - x for 0 <= x <= 1: with INTS on the integer units,
// too, else by the FP64 instructions.  The integer forms take some 40
// instructions for one, so they pay only where the FP64 pipe is the bound and
// their code runs from a loop: in the table kernel's curve and axis loops (512^2
// x 24 h: 1.557 -> 1.490 ms; everywhere in that kernel 1.586 ms; in the
// frontier's on-demand rows, which are bound by latency, 24.4 -> 26.7 ms).
__device__ __noinline__ double done_minus_any(double x) { return __dsub_rn(1.0, x); }
template <bool INTS>
__device__ __forceinline__ double dmul_pos(double x, double y) {
  if (!INTS) return __dmul_rn(x, y);
  return mid_range(bits_of(x)) && mid_range(bits_of(y)) ? mul_mid(x, y) : dmul_any(x, y);
}
template <bool INTS>
__device__ __forceinline__ double done_minus(double x) {
  if (!INTS) return __dsub_rn(1.0, x);
  return below_one(bits_of(x)) ? one_minus(x) : done_minus_any(x);
}
__device__ __forceinline__ double droot(double x) { return mid_range(bits_of(x)) ? sqrt_mid(x) : dsqrt_any(x); }

// a binary32 integer as binary64, by its bits
__device__ __forceinline__ double widen_int(float f) {
  const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
  return __hiloint2double(a ? (int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)) : 0, (int)(u << 29));
}

__device__ inline double dexp_series(double x) {
  // |x| < 704 (integer test of the high word) skips the range checks below
  if ((__double2hiint(x) & 0x7fffffff) >= 0x40860000) {
    if (x != x) return x;
    if (x > 709.78) return __longlong_as_double(0x7ff0000000000000LL);
    if (x < -745.2) return 0.0;
  }
  const double kd = rint(__dmul_rn(x, kInvLn2));
  const double r = __dsub_rn(__dsub_rn(x, __dmul_rn(kd, kLn2Hi)), __dmul_rn(kd, kLn2Lo));
  double p = g_mc.inv_fact[13];
#pragma unroll
  for (int i = 12; i >= 0; --i) p = __fma_rn(p, r, g_mc.inv_fact[i]);
  return scale2(p, (int)kd);
}

__device__ inline double dlog_series(double x) {
  int e = 0;
  const int hx = __double2hiint(x);
  if (hx < 0x00100000 || hx >= 0x7ff00000) {   // not a positive normal finite number
    if (x != x) return x;
    if (x < 0.0) return __longlong_as_double(0x7ff8000000000000LL);
    if (x == 0.0) return __longlong_as_double((long long)0xfff0000000000000ULL);
    if (__double_as_longlong(x) == 0x7ff0000000000000LL) return x;
    if (x < 0x1p-1022) { x = __dmul_rn(x, 0x1p54); e = -54; }
  }
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  e += (int)((b >> 52) & 0x7ff) - 1023;
  b = (b & 0x000fffffffffffffULL) | 0x3ff0000000000000ULL;
  double m = __longlong_as_double((long long)b);
  if (m > kSqrt2) { m = __dmul_rn(m, 0.5); e += 1; }
  const double f = __dsub_rn(m, 1.0);
  const double s = __ddiv_rn(f, __dadd_rn(2.0, f));
  const double z = __dmul_rn(s, s);
  double q = g_mc.log_c[10];
#pragma unroll
  for (int n = 9; n >= 1; --n) q = __fma_rn(q, z, g_mc.log_c[n]);
  const double s2 = __dadd_rn(s, s);
  const double lm = __fma_rn(__dmul_rn(s2, z), q, s2);
  const double ed = (double)e;
  return __dadd_rn(__dmul_rn(ed, kLn2Hi), __fma_rn(ed, kLn2Lo, lm));
}

// exp's argument reduction, |x| < 704: k = rint(RN(x 64/ln2)) and r = x - k
// ln2/64 by two fused steps.  k is found in binary32 off the FP64 pipe: x
// truncated to 24 bits and two roundings leave the product within 2^-21 of
// itself, so unless it lies that close to a half the nearest integer is the same.
__device__ __forceinline__ double exp_reduce(double x, int *k_out) {
  const uint32_t hx = (uint32_t)__double2hiint(x), ax = hx & 0x7fffffffu;
  const float xf = ax < 0x38100000u
      ? 0.0f : __uint_as_float((hx & 0x80000000u) | ((ax - 0x38000000u) << 3) | ((uint32_t)__double2loint(x) >> 29));
  const float t = __fmul_rn(xf, (float)(kInvLn2 * 64.0));
  const float s = __fadd_rn(t, 12582912.0f);   // 1.5 2^23: rounds to an integer, |t| < 2^17
  const float kf = __fsub_rn(s, 12582912.0f);
  int k = __float_as_int(s) - 0x4B400000;
  double kd = widen_int(kf);
  if (!(fabsf(__fsub_rn(t, kf)) < 0.4999f - fabsf(t) * 0x1p-21f)) {
    kd = drint_product(x, kInvLn2 * 64.0);
    k = (int)kd;
  }
  *k_out = k;
  return __fma_rn(-kd, kLn2Lo / 64.0, __fma_rn(-kd, kLn2Hi / 64.0, x));
}

// 2^(k/64) exp(r), r2 = RN(r r)
__device__ __forceinline__ double exp_finish(double r, double r2, int k) {
  bool exact;
  double q = exp_steps(r, &exact);
  if (!exact) q = exp_steps_any(r);
  const double p = __fma_rn(q, r2, r);   // exp(r) - 1 to r^5
  const double t = __ldg(&g_exp_tab[k & 63]);
  const double y = __fma_rn(t, p, t);                  // in [2^(-1/128), 2)
  const int m = k >> 6;
  // y 2^m is exact while it stays normal: add m to the exponent field
  if (m >= -1020 && m <= 1022) return __longlong_as_double(__double_as_longlong(y) + ((long long)m << 52));
  return dscale_any(y, m);
}

__device__ inline double dexp(double x) {
  if ((__double2hiint(x) & 0x7fffffff) >= 0x40860000) {   // |x| >= 704
    const double far = dexp_far(x);
    if (bits_of(far) != bits_of(1.0)) return far;
  }
  int k;
  const double r = exp_reduce(x, &k);
  return exp_finish(r, __dmul_rn(r, r), k);
}

// exp(x) and exp(-x) for 0 <= x < 704: the reduction is odd in x, so one serves both
__device__ __forceinline__ void dexp_both(double x, double *up, double *down) {
  int k;
  const double r = exp_reduce(x, &k);
  const double r2 = __dmul_rn(r, r);
  *up = exp_finish(r, r2, k);
  *down = exp_finish(-r, r2, -k);
}

// log of a positive normal x, e0 added to its exponent
__device__ __forceinline__ double dlog_normal(double x, int e0) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = e0 + (int)((b >> 52) & 0x7ff) - 1023;
  const int j = (int)((b >> 44) & 255);
  b = (b & 0x000fffffffffffffULL) | 0x3ff0000000000000ULL;
  const double m = __longlong_as_double((long long)b);
  const double r = __fma_rn(m, __ldg(&g_log_inv[j]), -1.0);
  // log(1 + r) = r - r^2/2 + r^3/3 - ... - r^6/6
  bool exact;
  double q = log_steps(r, &exact);
  if (!exact) q = log_steps_any(r);
  const double lp = __fma_rn(q, __dmul_rn(r, r), r);
  const double ed = widen_int((float)e);
  // e kLn2Hi is exact (11 and 29 bits), so the fused sum rounds once, as the separate one
  const double hi = __fma_rn(ed, kLn2Hi, __ldg(&g_log_tab[j]));
  const double lo = __fma_rn(ed, kLn2Lo, lp);
  return __dadd_rn(hi, lo);
}

// log of anything else
__device__ __noinline__ double dlog_any(double x) {
  if (x != x) return x;
  if (x < 0.0) return __longlong_as_double(0x7ff8000000000000LL);
  if (x == 0.0) return __longlong_as_double((long long)0xfff0000000000000ULL);
  if (__double_as_longlong(x) == 0x7ff0000000000000LL) return x;
  return dlog_normal(__dmul_rn(x, 0x1p54), -54);   // subnormal
}

__device__ inline double dlog(double x) {
  const int hx = __double2hiint(x);
  return hx < 0x00100000 || hx >= 0x7ff00000 ? dlog_any(x) : dlog_normal(x, 0);
}

__device__ inline double dpow(double x, double y) {
  if (x > 0.0) {
    const double y2 = __dadd_rn(y, y);
    if (y > 0.0 && y2 <= 16.0 && rint(y2) == y2) {   // y = n or n + 1/2, n <= 8
      const int n = (int)y;
      double r = 1.0;
      if (n > 0) {
        r = x;
        for (int i = 1; i < n; ++i) r = __dmul_rn(r, x);
      }
      if (((int)y2) & 1) r = (n > 0) ? __dmul_rn(r, __dsqrt_rn(x)) : __dsqrt_rn(x);
      return r;
    }
    return dexp(__dmul_rn(y, dlog(x)));
  }
  if (x == 0.0) return (y > 0.0) ? 0.0 : ((y == 0.0) ? 1.0 : __longlong_as_double(0x7ff0000000000000LL));
  return __longlong_as_double(0x7ff8000000000000LL);
}

// dpow with the exponent's kind decided ahead: n2 = 2y when y is a positive
// multiple of 1/2 up to 8 (the case dpow treats with products and a square
// root), else 0 -- the same results as dpow(x, y) without testing y
__device__ __noinline__ double dpow_any(double x, double y) {   // x not positive
  if (x == 0.0) return (y > 0.0) ? 0.0 : ((y == 0.0) ? 1.0 : __longlong_as_double(0x7ff0000000000000LL));
  return __longlong_as_double(0x7ff8000000000000LL);
}

template <bool INTS = false>
__device__ __forceinline__ double dpow_n2(double x, double y, int n2) {
  if (!pos(x)) return dpow_any(x, y);
  if (n2 == 0) return dexp(__dmul_rn(y, dlog(x)));
  const int n = n2 >> 1;
  double r = x;
#pragma unroll 1
  for (int i = 1; i < n; ++i) r = dmul_pos<INTS>(r, x);
  if (n2 & 1) {
    const double root = droot(x);
    r = n > 0 ? dmul_pos<INTS>(r, root) : root;
  }
  return r;
}

// host: n2 of dpow_n2 for a constant exponent
inline int pow_half_steps(double y) {
  const double y2 = y + y;
  return (y > 0.0 && y2 <= 16.0 && std::nearbyint(y2) == y2) ? (int)y2 : 0;
}

// fills g_exp_tab / g_log_inv / g_log_tab with the series forms (one block of 256)
__global__ void k_math_tables() {
  const int j = threadIdx.x;
  if (j < 64)
    g_exp_tab[j] = dexp_series(__dadd_rn(__dmul_rn((double)j, kLn2Hi / 64.0), __dmul_rn((double)j, kLn2Lo / 64.0)));
  if (j < 256) {
    const double v = __ddiv_rn(1.0, __dadd_rn(1.0, __ddiv_rn((double)j, 256.0)));
    g_log_inv[j] = v;
    g_log_tab[j] = -dlog_series(v);
  }
}

__device__ inline void dsincos_deg(double x, double *s_out, double *c_out) {
  const double qd = rint(__ddiv_rn(x, 90.0));
  const double r = __dsub_rn(x, __dmul_rn(qd, 90.0));
  const double t = __dmul_rn(r, kDeg2Rad);
  const double t2 = __dmul_rn(t, t);
  double ps = g_mc.sin_c[8];
#pragma unroll
  for (int n = 7; n >= 1; --n) ps = __fma_rn(ps, t2, g_mc.sin_c[n]);
  const double sn = __fma_rn(__dmul_rn(t, t2), ps, t);
  double pc = g_mc.cos_c[9];
#pragma unroll
  for (int n = 8; n >= 1; --n) pc = __fma_rn(pc, t2, g_mc.cos_c[n]);
  const double cs = __fma_rn(t2, pc, 1.0);
  const long long qi = (long long)qd;
  const int q = (int)(((qi % 4) + 4) % 4);
  double s, c;
  if (q == 0) { s = sn; c = cs; }
  else if (q == 1) { s = cs; c = -sn; }
  else if (q == 2) { s = -sn; c = -cs; }
  else { s = -cs; c = sn; }
  *s_out = s;
  *c_out = c;
}

// ---------------------------------------------------------------- binary32
__device__ __forceinline__ float pow2if(int k) {  // exact 2^k, -126 <= k <= 127
  return __int_as_float((k + 127) << 23);
}

__device__ __forceinline__ float scale2f(float p, int k) {
  if (k > 127) return __fmul_rn(__fmul_rn(p, pow2if(127)), pow2if(k - 127));
  if (k < -126) return __fmul_rn(__fmul_rn(p, pow2if(k + 64)), pow2if(-64));
  return __fmul_rn(p, pow2if(k));
}

__device__ inline float fexp(float x) {
  if (x != x) return x;
  if (x > 88.72f) return __int_as_float(0x7f800000);
  if (x < -103.9f) return 0.0f;
  const float kf = rintf(__fmul_rn(x, kInvLn2F));
  const float r = __fsub_rn(__fsub_rn(x, __fmul_rn(kf, kLn2HiF)), __fmul_rn(kf, kLn2LoF));
  float p = g_mc.inv_fact_f[7];
#pragma unroll
  for (int i = 6; i >= 0; --i) p = __fmaf_rn(p, r, g_mc.inv_fact_f[i]);
  return scale2f(p, (int)kf);
}

__device__ inline float flog(float x) {
  if (x != x) return x;
  if (x < 0.0f) return __int_as_float(0x7fc00000);
  if (x == 0.0f) return __int_as_float((int)0xff800000u);
  if (__float_as_int(x) == 0x7f800000) return x;
  int e = 0;
  if (x < 0x1p-126f) { x = __fmul_rn(x, 0x1p24f); e = -24; }
  unsigned int b = (unsigned int)__float_as_int(x);
  e += (int)((b >> 23) & 0xff) - 127;
  b = (b & 0x007fffffu) | 0x3f800000u;
  float m = __int_as_float((int)b);
  if (m > kSqrt2F) { m = __fmul_rn(m, 0.5f); e += 1; }
  const float f = __fsub_rn(m, 1.0f);
  const float s = __fdiv_rn(f, __fadd_rn(2.0f, f));
  const float z = __fmul_rn(s, s);
  float q = g_mc.log_cf[5];
#pragma unroll
  for (int n = 4; n >= 1; --n) q = __fmaf_rn(q, z, g_mc.log_cf[n]);
  const float s2 = __fadd_rn(s, s);
  const float lm = __fmaf_rn(__fmul_rn(s2, z), q, s2);
  const float ef = (float)e;
  return __fadd_rn(__fmul_rn(ef, kLn2HiF), __fmaf_rn(ef, kLn2LoF, lm));
}

// flog for u in [2^-25, 1) and fexp for |x| < 64 ln 2: the same arithmetic
// without the special-value branches (NaN, sign, zero, infinity, subnormal,
// overflow, underflow) that such arguments never take; the perturbation's
// draws always lie in these ranges
__device__ __forceinline__ float flog_unit(float x) {
  const unsigned int b0 = (unsigned int)__float_as_int(x);
  int e = (int)((b0 >> 23) & 0xff) - 127;
  float m = __int_as_float((int)((b0 & 0x007fffffu) | 0x3f800000u));
  if (m > kSqrt2F) { m = __fmul_rn(m, 0.5f); e += 1; }
  const float f = __fsub_rn(m, 1.0f);
  const float s = __fdiv_rn(f, __fadd_rn(2.0f, f));
  const float z = __fmul_rn(s, s);
  float q = g_mc.log_cf[5];
#pragma unroll
  for (int n = 4; n >= 1; --n) q = __fmaf_rn(q, z, g_mc.log_cf[n]);
  const float s2 = __fadd_rn(s, s);
  const float lm = __fmaf_rn(__fmul_rn(s2, z), q, s2);
  const float ef = (float)e;
  return __fadd_rn(__fmul_rn(ef, kLn2HiF), __fmaf_rn(ef, kLn2LoF, lm));
}

__device__ __forceinline__ float fexp_small(float x) {
  const float kf = rintf(__fmul_rn(x, kInvLn2F));
  const float r = __fsub_rn(__fsub_rn(x, __fmul_rn(kf, kLn2HiF)), __fmul_rn(kf, kLn2LoF));
  float p = g_mc.inv_fact_f[7];
#pragma unroll
  for (int i = 6; i >= 0; --i) p = __fmaf_rn(p, r, g_mc.inv_fact_f[i]);
  return __fmul_rn(p, pow2if((int)kf));
}

// cos(2 pi u)
__device__ inline float fcos_turns(float u) {
  const float qf = rintf(__fmul_rn(u, 4.0f));
  const float r = __fsub_rn(u, __fmul_rn(qf, 0.25f));
  const float t = __fmul_rn(r, kTwoPiF);
  const float t2 = __fmul_rn(t, t);
  float ps = g_mc.sin_cf[4];
#pragma unroll
  for (int n = 3; n >= 1; --n) ps = __fmaf_rn(ps, t2, g_mc.sin_cf[n]);
  const float sn = __fmaf_rn(__fmul_rn(t, t2), ps, t);
  float pc = g_mc.cos_cf[5];
#pragma unroll
  for (int n = 4; n >= 1; --n) pc = __fmaf_rn(pc, t2, g_mc.cos_cf[n]);
  const float cs = __fmaf_rn(t2, pc, 1.0f);
  const int q = (int)qf & 3;   // quadrants 0..3: cs, -sn, -cs, sn
  const float v = (q & 1) ? sn : cs;
  return __int_as_float(__float_as_int(v) ^ (((q + 1) & 2) << 30));
}

// ---------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon et al., SC'11): 10 rounds, Weyl key schedule.
struct U4 { uint32_t x, y, z, w; };

// (Two rounds to a loop turn: all ten unrolled run 2 % faster alone and 6 %
// slower in a frontier with several warps on a scheduler, by instruction fetches.)
__device__ __forceinline__ U4 philox4x32_10(U4 c, uint32_t k0, uint32_t k1) {
#pragma unroll 2
  for (int round = 0; round < 10; ++round) {
    if (round > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
  }
  return c;
}

// Multiplicative ROS perturbation of (replica, cell, hour): f = exp(sigma z),
// z ~ N(0,1) by Box-Muller from the Philox block at counter
// (replica, cell, hour, 0) under the run key; binary32; sigma == 0 -> 1.
__device__ inline float noise_factor(uint64_t seed, uint32_t replica, uint32_t cell,
                                     uint32_t hour, float sigma) {
  if (sigma == 0.0f) return 1.0f;
  const U4 x = philox4x32_10(U4{replica, cell, hour, 0u}, (uint32_t)seed,
                             (uint32_t)(seed >> 32));
  const float u1 = __fmul_rn(__fadd_rn((float)(x.x >> 8), 0.5f), 0x1p-24f);
  const float u2 = __fmul_rn(__fadd_rn((float)(x.y >> 8), 0.5f), 0x1p-24f);
  // u1 >= 2^-25, so |z| <= sqrt(50 ln 2) < 6 and |sigma z| < 6 for sigma <= 1
  const float z = __fmul_rn(__fsqrt_rn(__fmul_rn(-2.0f, flog_unit(u1))), fcos_turns(u2));
  return fexp_small(__fmul_rn(sigma, z));
}

// the perturbation as a 32.32 fixed-point multiplier f 2^32: exact, since
// f >= 2^-9 has a binary32 significand whose scaled value is an integer.  Built
// from the bits (significand shifted by the exponent) rather than by a
// float-to-int64 conversion, which is slow on this GPU.
__device__ __forceinline__ uint64_t noise_fixed(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint64_t m = (uint64_t)((b & 0x7FFFFFu) | 0x800000u);
  return m << ((int)(b >> 23) - 118);   // 2^(e - 127 - 23 + 32), e >= 118 for f >= 2^-9
}

// per-period increment (base * F + 2^31) >> 32, capped at the axis length dk <
// 2^53, for 2^23 <= F < 2^41, from the 32-bit halves: with base = b1 2^32 + b0
// and F = f1 2^32 + f0 it is b1 f1 2^32 + b1 f0 + b0 f1 + ((b0 f0 + 2^31) >> 32).
// base >= 2^62 or b1 f1 >= 2^21 alone exceeds any dk; otherwise the sum stays
// below 2^63
__device__ __forceinline__ int64_t apply_noise(int64_t base, uint64_t F, int64_t dk) {
  const uint32_t b0 = (uint32_t)base, b1 = (uint32_t)((uint64_t)base >> 32);
  const uint32_t f0 = (uint32_t)F, f1 = (uint32_t)(F >> 32);
  const uint64_t top = (uint64_t)b1 * f1;
  if ((top >> 21) | (b1 >> 30)) return dk;
  const uint64_t inc = (top << 32) + (uint64_t)b1 * f0 + (uint64_t)b0 * f1 + (((uint64_t)b0 * f0 + 0x80000000ull) >> 32);
  return inc > (uint64_t)dk ? dk : (int64_t)inc;
}

}  // namespace c2f
