// FP64 division, reciprocal and square root with few FP64-pipe operations, and
// comparisons and halves without any, for GB300's scarce FP64 pipe.
#pragma once
#include <math.h>
#include <stdint.h>

namespace wcns {

// CUDA's division and square root, out of line: they serve rare operands, and
// inlined at every use they made up a quarter of the sweeps' code (a 2D sweep
// 228 -> 176 KB, 155 KB with the limiter certification as loops), which then
// did not fit the instruction caches: with the interpolation's two sides as
// one loop body as well, 2048 x 1024 8.67 -> 8.15 ms, 120^3 18.9 -> 16.1 ms.
static __device__ __noinline__ double div_ieee(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt_ieee(double a) { return sqrt(a); }

// Mantissa of a normal FP64 value as an FP32 pair in [1, 2): h the leading 24
// bits, l the rest.
__device__ __forceinline__ void mantissa2(unsigned long long u, float &h, float &l) {
  h = __uint_as_float(0x3F800000u | (unsigned int)((u >> 29) & 0x7FFFFFull));
  l = (float)((unsigned int)u & 0x1FFFFFFFu) * 2.220446049250313e-16f;
}
// (r + d) 2^(f - 1022) as FP64 bits, for an FP32 r in [0.5, 1) and a
// correction |d| < 2^-21 r; d enters to 2^-50.
__device__ __forceinline__ double seed64(float r, float d, unsigned int f) {
  const unsigned int m = __float_as_uint(r) & 0x7FFFFFu;
  const long long di = __float2int_rn(d * 1125899906842624.0f);
  return __longlong_as_double((((long long)f << 52) | ((long long)m << 29)) + (di << 3));
}
// 1/|b| to a relative error below 2^-43 for a normal b below 2^1021 in
// magnitude (eb its exponent field), without FP64 operations: the
// approximate FP32 reciprocal of the mantissa and one Newton-Raphson
// correction in FP32, packed with integer operations.
__device__ __forceinline__ double rcp_seed(unsigned long long ub, unsigned int eb) {
  float h, l, r;
  mantissa2(ub, h, l);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h));
  r = fminf(fmaxf(r, 0.5f), 0.99999994f);
  const float e = fmaf(-l, r, fmaf(-h, r, 1.0f));
  return seed64(r, r * e, 2045u - eb);
}

// a / b in FP64 with three FP64-pipe operations (the FP64 pipe is GB300's
// scarce one; an IEEE division takes about nine): y from rcp_seed, the
// quotient q0 = a y, and one correction q1 = q0 + y (a - b q0) with the
// remainder from a fused multiply-add (Markstein, IBM J. Res. Dev. 34 (1990)
// 111), which leaves q1 within one unit in the last place of a / b.  With the
// reciprocal refined in FP64 (two operations more) and CUDA's square roots a
// 2048 x 1024 step took 11.05 ms instead of 10.35.  Operands
// outside the range where that holds (b zero, subnormal, not finite or above
// 2^1021; a not finite or below 2^-959, where the remainder would underflow;
// a / b near the overflow threshold) take the IEEE division, except a zero
// numerator over a finite nonzero b, whose quotient is the signed zero a * b.
__device__ __forceinline__ double div_nr(double a, double b) {
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b);
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
  const unsigned int eb = (unsigned int)(ub >> 52) & 0x7FFu;
  const unsigned int ea = (unsigned int)(ua >> 52) & 0x7FFu;
  if (eb - 1u >= 2044u || ea - 64u >= 1983u || (int)ea - (int)eb > 1020) {
    if ((ua << 1) == 0 && (ub << 1) != 0 && eb != 0x7FFu) return a * b;
    return div_ieee(a, b);
  }
  const double y = __longlong_as_double(__double_as_longlong(rcp_seed(ub, eb)) | (long long)(ub & 0x8000000000000000ull));
  const double q0 = __dmul_rn(a, y);
  return fma(y, fma(-b, q0, a), q0);
}
// 1 / b: two FP64-pipe operations, within 0.51 units in the last place
__device__ __forceinline__ double rcp_nr(double b) {
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b);
  const unsigned int eb = (unsigned int)(ub >> 52) & 0x7FFu;
  if (eb - 1u >= 2044u) return div_ieee(1.0, b);
  const double y = __longlong_as_double(__double_as_longlong(rcp_seed(ub, eb)) | (long long)(ub & 0x8000000000000000ull));
  return fma(y, fma(-b, y, 1.0), y);
}
// 1/sqrt(t) to a relative error below 2^-43 for a normal positive t, as
// rcp_seed forms the reciprocal.
__device__ __forceinline__ double rsqrt_seed(double t) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(t);
  const int e = (int)(u >> 52) - 1023, odd = e & 1;
  float h, l, r;
  mantissa2(u, h, l);
  const float two = odd ? 2.0f : 1.0f;
  h *= two;
  l *= two;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h));
  r = fminf(fmaxf(r, 0.5f), 0.99999994f);
  const float q = r * r, qe = fmaf(r, r, -q);
  const float d = fmaf(-l, q, fmaf(-h, qe, fmaf(-h, q, 1.0f)));
  return seed64(r, r * fmaf(0.375f * d, d, 0.5f * d), (unsigned int)(1022 - ((e - odd) >> 1)));
}
// Order of two values without an FP64-pipe compare (sign-magnitude bits as
// integers; a NaN orders beyond the infinities).
__device__ __forceinline__ bool less64(double a, double b) {
  long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  x ^= (long long)((unsigned long long)(x >> 63) >> 1);
  y ^= (long long)((unsigned long long)(y >> 63) >> 1);
  return x < y;
}
// 0.5 x: an exponent decrement wherever the result is normal
__device__ __forceinline__ double half64(double x) {
  const unsigned int e = ((unsigned int)__double2hiint(x) >> 20) & 0x7FFu;
  return e - 2u < 0x7FDu ? __longlong_as_double(__double_as_longlong(x) - (1ll << 52)) : 0.5 * x;
}
// Half of a normal value (an exponent decrement).
__device__ __forceinline__ double half_normal(double x) {
  return __longlong_as_double(__double_as_longlong(x) - (1ll << 52));
}
// sqrt(t): three FP64-pipe operations, within 0.51 units in the last place;
// CUDA's square root outside the seed's range.
__device__ __forceinline__ double sqrt_nr(double t) {
  const unsigned int hi = (unsigned int)__double2hiint(t);
  if (hi - 0x10000000u >= 0x60000000u) return sqrt_ieee(t);  // not in [2^-767, 2^769)
  const double y = rsqrt_seed(t), g = __dmul_rn(t, y);
  return fma(fma(-g, g, t), half_normal(y), g);
}
// sqrt(n / d): five FP64-pipe operations (a Newton-Raphson step on
// c^2 d = n from c = n rsqrt(n d)), within 1.01 units in the last place: c d
// is rounded before the remainder.
__device__ __forceinline__ double sqrt_ratio(double n, double d) {
  const unsigned int hn = (unsigned int)__double2hiint(n), hd = (unsigned int)__double2hiint(d);
  // both in [2^-447, 2^449)
  if (hn - 0x24000000u >= 0x38000000u || hd - 0x24000000u >= 0x38000000u) return sqrt_ieee(div_ieee(n, d));
  const double y = rsqrt_seed(__dmul_rn(n, d)), c = __dmul_rn(n, y);
  return fma(fma(-c, __dmul_rn(c, d), n), half_normal(y), c);
}

// A product kept apart from a following sum.  The compiler may contract
// a * b + c * d either way, and differently in two kernels that share the
// code: wherever a sum has two products, or a product several uses, the FP64
// code says which one is fused, so that a batched problem and the same
// problem on its own grid stay bit for bit equal.
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }

// FP32 image of an FP64 value from its high word alone (integer operations
// only): sign, exponent and the leading 20 mantissa bits, truncated toward
// zero, so |x - t(x)| < 2^-20 |x| and |t(x)| <= |x|.  A value below the
// FP32 normal range maps to 0 (absolute error below 2^-126: the bounds below
// add CTINY for it); a value at or above 2^128 or not finite maps to a NaN,
// which fails every certification test.
__device__ __forceinline__ float trunc32(double x) {
  const unsigned int hi = (unsigned int)__double2hiint(x);
  const unsigned int mag = hi & 0x7FFFFFFFu;
  // FP64 exponent field in [897, 1150] <=> FP32 exponent field in [1, 254]
  if (mag - 0x38100000u < 0x0FE00000u) return __uint_as_float((hi & 0x80000000u) | ((mag - 0x38000000u) << 3));
  return mag < 0x38100000u ? 0.0f : __uint_as_float(0x7FC00000u);
}

}  // namespace wcns
