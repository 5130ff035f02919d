// WCNS-IS interpolation (Sec. 4.3) of FP64 deviations without FP64
// arithmetic.
//
// Why: an FP64 warp instruction occupies an SM's FP64 units for 16 cycles on
// GB300, an FP32 or integer one its 128 lanes for a quarter to half a cycle,
// and the interpolation's ~65 operations a value were 70 % of the FP64
// sweeps' FP64 work (1034 to 1110 add/mul/fma per cell and direction before,
// about 380 after: 27.4 against 11.0 ms a step of the 2048 x 1024
// shock/bubble run, 43.6 against 22.2 ms of a 120^3 bubble collapse).
//
// How: the interpolated value is the linear fifth-order one plus a correction
// by the nonlinear weights,
//   u = u_lin + sum_k d_k rho_k (s_k - u_lin) / (1 + sum_k d_k rho_k),
//   rho_0 = tau^2 / (b0 b01), rho_1 = tau^2 / (b1 b01), rho_{2,3} = tau / b_{2,3}
// (d_k the linear weights, b_k = beta_k + eps, s_k the sub-stencil values).
// - The five deviations become integers on a common binary scale, cut at
//   2^-54 of the largest one's binade; u_lin, s_k - u_lin and every difference
//   in the indicators are exact from there.
// - The correction is formed in FP32, relative error below 2^-19, and where
//   that is not enough in pairs of FP32 values, below 2^-39; both errors are
//   bounded by S = sum d_k rho_k |s_k - u_lin| / (1 + sum d_k rho_k).
// - A value is accepted where the bound is at most 2^-54 (scale + |u|).  With
//   the cut (1.4 times 2^-54 of the largest deviation's binade through u_lin,
//   and as much again through the weights) the result is within about
//   2^-52 (scale + |u|), at worst; in the root mean square the sum scale + u
//   that the caller forms is as accurate as from the formula in FP64.
//   Elsewhere (strong jumps of the field inside the stencil) the caller
//   evaluates the printed formula in FP64.
// Every decision depends on the value's own stencil only.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define WISW __host__ __device__ __forceinline__
#else
#define WISW static inline
#endif
#ifdef __CUDA_ARCH__
#define WISW_ROLLED _Pragma("unroll 1")
#else
#define WISW_ROLLED
#endif

namespace wcns {
namespace isw {

// --- bit-level helpers (device intrinsics; plain C++ on the host) ----------
WISW unsigned hi32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return (unsigned)(u >> 32);
#endif
}
WISW unsigned lo32(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return (unsigned)u;
#endif
}
WISW double from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
WISW float from_bits32(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  memcpy(&x, &u, 4);
  return x;
#endif
}
WISW int clz32(unsigned u) {
#ifdef __CUDA_ARCH__
  return __clz((int)u);
#else
  return u ? __builtin_clz(u) : 32;
#endif
}
WISW float frcp(float b) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  return r;
#else
  return 1.0f / b;
#endif
}
WISW float fdiv(float a, float b) { return a * frcp(b); }
WISW float frsqrt(float b) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  return r;
#else
  return 1.0f / sqrtf(b);
#endif
}
WISW int frint(float x) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)nearbyintf(x);
#endif
}

// --- fixed point -----------------------------------------------------------
// x as an integer multiple of 2^-54 of the binade top above exponent field
// E (|x| < 2^(E - 1022)), truncated toward zero: |fix| < 2^54.  Zeros and
// subnormals give 0.
WISW int64_t fix(double x, int E) {
  const unsigned h = hi32(x), l = lo32(x);
  const int e = (int)((h >> 20) & 0x7FFu);
  const unsigned m = (h & 0xFFFFFu) | 0x100000u;
  const uint64_t f = ((((uint64_t)m << 32) | l) << 1);
  const int s = E - e;
  const int64_t v = (s < 64 && e != 0) ? (int64_t)(f >> s) : 0;
  return (int)h < 0 ? -v : v;
}
// v 2^(E - 1022 - 61) rounded to nearest FP64 (|v| < 2^63, 64 <= E <= 2040).
WISW double unfix(int64_t v, int E) {
  if (v == 0) return 0.0;
  const uint64_t sgn = (uint64_t)(v >> 63);
  uint64_t a = ((uint64_t)v ^ sgn) - sgn;
  const unsigned ah = (unsigned)(a >> 32);
  const int n = ah ? clz32(ah) : 32 + clz32((unsigned)a);
  a <<= n;  // leading bit at 2^63
  const uint64_t m = (a >> 11) + ((a >> 10) & 1u);
  return from_bits((sgn << 63) + ((uint64_t)(unsigned)(E + 2 - n) << 52) + m);
}
// v / 2^32 in FP32, relative error below 2^-23 plus 2^-24 absolute
// (|v| <= 2^56)
WISW float fx(int64_t v) {
  return fmaf((float)((unsigned)v >> 8), 5.9604644775390625e-08f, (float)(int)(v >> 32));
}

// x as an integer multiple of 2^-62 of the binade top above E, truncated
WISW int64_t fix62(double x, int E) {
  const unsigned h = hi32(x), l = lo32(x);
  const int e = (int)((h >> 20) & 0x7FFu);
  const unsigned m = (h & 0xFFFFFu) | 0x100000u;
  const uint64_t f = ((((uint64_t)m << 32) | l) << 9);
  const int s = E - e;
  const int64_t v = (s < 64 && e != 0) ? (int64_t)(f >> s) : 0;
  return (int)h < 0 ? -v : v;
}
WISW unsigned umax(unsigned a, unsigned b) { return a > b ? a : b; }
WISW unsigned mag32(double x) { return hi32(x) & 0x7FFFFFFFu; }

// The linear combination of the HCS reconstruction (Sec. 4.1),
//   2100 (G^ - g~) = 972 g~ - 505 (g0 + g1) + 20 (gm1 + g2) - (gm2 + g3),
// exact on the values' common scale (2^-62 of the largest; rounded to nearest
// FP64 at the end): false where their exponents leave the range.
WISW bool hcs_correction(double gt, double gm2, double gm1, double g0, double g1, double g2, double g3, double &c) {
  const unsigned mx = umax(umax(umax(mag32(gt), mag32(gm2)), umax(mag32(gm1), mag32(g0))),
                           umax(umax(mag32(g1), mag32(g2)), mag32(g3)));
  const int E = (int)(mx >> 20);
  c = 0.0;
  if (E < 128 || E > 1900) return mx == 0;
  const int64_t t = fix62(gt, E), a = fix62(gm2, E), b = fix62(gm1, E), p = fix62(g0, E), q = fix62(g1, E),
                d = fix62(g2, E), f = fix62(g3, E);
  // 32-bit halves: |high| <= 2^30, so every sum below stays inside 64 bits
  const auto H = [](int64_t v) { return (int64_t)(int)(v >> 32); };
  const auto L = [](int64_t v) { return (int64_t)(unsigned)v; };
  const int64_t lo = 972 * L(t) - 505 * (L(p) + L(q)) + 20 * (L(b) + L(d)) - (L(a) + L(f));
  const int64_t hi = 972 * H(t) - 505 * (H(p) + H(q)) + 20 * (H(b) + H(d)) - (H(a) + H(f)) + (lo >> 32);
  c = unfix((hi << 20) | (int64_t)((unsigned)lo >> 12), E + 11);
  return true;
}

// --- FP32 pairs ------------------------------------------------------------
struct F2 {
  float h, l;
};
WISW F2 fx2(int64_t v) {
  const float a = (float)(int)(v >> 32), b = (float)((unsigned)v >> 8) * 5.9604644775390625e-08f;
  const float s = a + b;
  return {s, b - (s - a)};
}
WISW F2 mul(F2 a, F2 b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  return {p, e};
}
WISW F2 sqr(F2 a) {
  const float p = a.h * a.h;
  return {p, fmaf(a.h + a.h, a.l, fmaf(a.h, a.h, -p))};
}
WISW F2 scale(F2 a, float s) { return {a.h * s, a.l * s}; }  // s a power of two
WISW F2 add(F2 a, F2 b) {
  const float s = a.h + b.h, t = s - a.h;
  const float e = (a.h - (s - t)) + (b.h - t);
  return {s, e + (a.l + b.l)};
}
// a / b
WISW F2 div(F2 a, F2 b) {
  const float r = frcp(b.h), q = a.h * r;
  const float d = fmaf(-q, b.l, fmaf(-q, b.h, a.h) + a.l);
  return {q, d * r};
}

// One side's stencil in integers: the differences around the upwind node.
//   d0 = u_{i+1} - u_i, dm the difference on the far side of the upwind node,
//   Da, Db, Dc second differences at the node behind the upwind node, at it,
//   and at the downwind one; c* the first-difference parts of the indicators.
struct Side {
  int64_t dm, Da, Db, Dc, c01, c2, c3;
};

constexpr float K133 = 13.0f / 3.0f;
constexpr float K133L = (float)(13.0 / 3.0 - (double)K133);
constexpr float UNIT = 4194304.0f;  // 2^22: the FP32 image of the largest |U|
constexpr float FLOORB = 256.0f;    // 2^-36 UNIT^2: smallest indicator taken as is

struct E4 {
  int64_t e0, e1, e2, e3;  // 128 (s_k - u_lin)
};
WISW E4 offsets(const Side &s) {
  const int64_t m = 3 * s.Da;
  E4 e;
  e.e0 = 5 * s.Dc - m + (s.Db << 4) - (s.Db << 1);
  e.e1 = e.e0 - (s.Db << 6);
  e.e2 = e.e0 - (s.Dc << 4);
  e.e3 = e.e1 + (m << 4);
  return e;
}

// FP32 evaluation: the weighted correction 128 (u - u_lin) in units of 2^39,
// and the bounds' ingredients.
struct Est {
  float corr, S, G, minb, mint, flr;
};
WISW Est side32(const Side &s, const E4 &e, float d0, float eps) {
  const float dm = fx(s.dm), Da = fx(s.Da), Db = fx(s.Db), Dc = fx(s.Dc);
  const float c01 = fx(s.c01), c2 = fx(s.c2 >> 2), c3 = fx(s.c3 >> 2);
  const float ta = fx((s.Da - 2 * s.Db + s.Dc) >> 2), tc = fx((s.Da - s.Dc) >> 2);
  const float b0 = fmaf(4.0f * d0, d0, eps), b1 = fmaf(4.0f * dm, dm, eps);
  const float b01 = fmaf(K133 * Db, Db, fmaf(c01, c01, eps));
  const float b2 = fmaf(K133 * Dc, Dc, fmaf(16.0f * c2, c2, eps));
  const float b3 = fmaf(K133 * Da, Da, fmaf(16.0f * c3, c3, eps));
  const float tau = 16.0f * fmaf(K133 * ta, ta, tc * tc);
  Est r;
  r.minb = fminf(fminf(fminf(b0, b1), fminf(b2, b3)), b01);
  r.mint = fminf(r.minb, fmaxf(tau, 1.4551915228366852e-11f));  // 2^-36
  r.flr = 0.0f;
  if (r.minb < FLOORB) {
    // Indicators below FLOORB: taken as FLOORB.  Where they are exact zeros,
    // and every other indicator and tau at least 2^16 FLOORB, their
    // sub-stencils carry the result up to 2^-14 either way.
    const float big = 65536.0f * FLOORB;
    const auto fine = [&](float b) { return b <= eps || b >= big; };
    r.flr = fine(b0) && fine(b1) && fine(b01) && fine(b2) && fine(b3) && (tau >= big || tau == 0.0f)
                ? 9.765625e-4f * UNIT : 16.0f * UNIT;
  }
  const float r01 = fdiv(tau, fmaxf(b01, FLOORB));
  const float w0 = 15.0f * fdiv(tau, fmaxf(b0, FLOORB)) * r01;
  const float w1 = 5.0f * fdiv(tau, fmaxf(b1, FLOORB)) * r01;
  const float w2 = 10.0f * fdiv(tau, fmaxf(b2, FLOORB));
  const float w3 = 2.0f * fdiv(tau, fmaxf(b3, FLOORB));
  const float g = (w0 + w1) + (w2 + w3);
  const float inv = frcp(32.0f + g);
  const float a0 = w0 * fx(e.e0 >> 7), a1 = w1 * fx(e.e1 >> 7), a2 = w2 * fx(e.e2 >> 7), a3 = w3 * fx(e.e3 >> 7);
  r.corr = ((a0 + a1) + (a2 + a3)) * inv;
  r.S = ((fabsf(a0) + fabsf(a1)) + (fabsf(a2) + fabsf(a3))) * inv;
  r.G = g * inv;
  return r;
}

// The same correction in FP32 pairs.
WISW F2 side2(const Side &s, const E4 &e, int64_t d0, F2 eps, bool use_eps) {
  const F2 K = {K133, K133L};
  F2 b0 = scale(sqr(fx2(d0)), 4.0f), b1 = scale(sqr(fx2(s.dm)), 4.0f);
  F2 b01 = add(sqr(fx2(s.c01)), mul(K, sqr(fx2(s.Db))));
  F2 b2 = add(scale(sqr(fx2(s.c2 >> 2)), 16.0f), mul(K, sqr(fx2(s.Dc))));
  F2 b3 = add(scale(sqr(fx2(s.c3 >> 2)), 16.0f), mul(K, sqr(fx2(s.Da))));
  const F2 tau = scale(add(mul(K, sqr(fx2((s.Da - 2 * s.Db + s.Dc) >> 2))), sqr(fx2((s.Da - s.Dc) >> 2))), 16.0f);
  if (use_eps) {
    b0 = add(b0, eps);
    b1 = add(b1, eps);
    b01 = add(b01, eps);
    b2 = add(b2, eps);
    b3 = add(b3, eps);
  }
  const F2 r01 = div(tau, b01);
  F2 w0 = mul(div(tau, b0), r01), w1 = mul(div(tau, b1), r01), w2 = div(tau, b2), w3 = div(tau, b3);
  // 15, 5, 10, 2 times: exact in the pair up to the rounding of the products
  w0 = mul(w0, {15.0f, 0.0f});
  w1 = mul(w1, {5.0f, 0.0f});
  w2 = mul(w2, {10.0f, 0.0f});
  w3 = scale(w3, 2.0f);
  const F2 den = add(add(add(w0, w1), add(w2, w3)), {32.0f, 0.0f});
  const F2 num = add(add(mul(w0, fx2(e.e0 >> 7)), mul(w1, fx2(e.e1 >> 7))),
                     add(mul(w2, fx2(e.e2 >> 7)), mul(w3, fx2(e.e3 >> 7))));
  return div(num, den);
}

// c (in units of 2^39) as an integer, to a unit: 2^-61 of the largest input.
// (Cut at 2^9 units, the two parts' roundings came to 2^-53 of the largest
// input, five times the rounding error of the FP64 formula for a field whose
// deviations are as large as its values.)
WISW int64_t corr_int(F2 c) {
  const int i1 = frint(c.h);
  const float g = (c.h - (float)i1) * 2147483648.0f;  // in units of 2^8
  const int i2 = frint(g);
  const float t = fmaf(c.l, 2147483648.0f, g - (float)i2);
  const int i3 = frint(t);
  return ((int64_t)i1 << 39) + (((int64_t)i2 + (int64_t)i3) << 8) + frint((t - (float)i3) * 256.0f);
}

// WCNS-IS of the deviations um2, um1, (0), up1, up2, up3 of nodes i-2 .. i+3
// from node i: left-biased value ul and right-biased value ur at i+1/2.
// e4: 4 eps.  scale: the magnitude whose rounding the result may carry: scl,
// and own times the largest deviation's binade / UNIT.
// Bit 0 / 1 set: ul / ur is within 2^-54 (scale + |u|) of the exact value
// plus the fixed-point rounding; clear: not decided.  bit 2: pairs used.
WISW int interpolate(double um2, double um1, double up1, double up2, double up3, double e4, float scl, double &ul,
                     double &ur, float own = 0.0f) {
  unsigned mx = hi32(um2) & 0x7FFFFFFFu, t;
  t = hi32(um1) & 0x7FFFFFFFu;
  mx = t > mx ? t : mx;
  t = hi32(up1) & 0x7FFFFFFFu;
  mx = t > mx ? t : mx;
  t = hi32(up2) & 0x7FFFFFFFu;
  mx = t > mx ? t : mx;
  t = hi32(up3) & 0x7FFFFFFFu;
  mx = t > mx ? t : mx;
  const int E = (int)(mx >> 20);
  ul = ur = 0.0;
  if (E < 64 || E > 2040) return mx == 0 ? 3 : 0;  // zeros; or outside the range below
  const int64_t X0 = fix(um2, E), X1 = fix(um1, E), X3 = fix(up1, E), X4 = fix(up2, E), X5 = fix(up3, E);
  const int64_t dm2 = X1 - X0, dm1 = -X1, d1 = X4 - X3, d2 = X5 - X4;
  const int64_t Dm = dm1 - dm2, D0 = X3 - dm1, D1 = d1 - X3, D2 = d2 - d1;
  // 4 eps in units of (2^(E-1022) / 2^22)^2 and the scale in units of
  // 2^(E-1022) / 2^22, exponents clamped to FP32's range (a larger eps
  // only lowers the already negligible weights; a smaller scale is safe)
  const unsigned eh = hi32(e4);
  int ee = (int)(eh >> 20) - 1023 - 2 * (E - 1022) + 44;
  ee = ee > 100 ? 100 : ee;
  const float eps = ee < -100 ? 0.0f : from_bits32(((unsigned)(ee + 127) << 23) | ((eh & 0xFFFFFu) << 3) | (lo32(e4) >> 29));
  int es = 1022 - E + 22;
  es = es > 100 ? 100 : (es < -120 ? -120 : es);
  const float sc = fmaf(scl, from_bits32((unsigned)(es + 127) << 23), own);
  const float mtol = 2.3283064365386963e-10f;  // 2^-54 UNIT
  int ret = 0;
  // one loop body for the two sides: unrolled, the code's fetch cost 8 % of a
  // 120^3 step (16.1 -> 17.5 ms)
  WISW_ROLLED
  for (int side = 0; side < 2; ++side) {
    const int64_t da = side ? d1 : dm1, db = side ? dm1 : d1;
    const Side s = {da, side ? D2 : Dm, side ? D1 : D0, side ? D0 : D1, da + X3, 3 * X3 - db, 3 * da - (side ? d2 : dm2)};
    const E4 e = offsets(s);
    const Est a = side32(s, e, fx(X3), eps);
    const int64_t lin = (X3 << 6) - e.e0;
    // what the result may be off by: 2^-54 (scale + |u|)
    const float tol = 5.551115123125783e-17f * (sc + fabsf(fx(lin >> 7) + a.corr));
    const float x = 1.9073486328125e-06f * frsqrt(a.mint);  // 2^-19 /
    const bool base = tol >= mtol;
    F2 c = {a.corr, 0.0f};
    if (base && a.S * (1.9073486328125e-06f + x) + a.flr <= tol) {
      ret |= 1 << side;
    } else if (base && a.minb >= FLOORB && a.S * (4.547473508864641e-13f + x) + 2.384185791015625e-07f * a.G <= tol) {
      const F2 ep = {eps, eps == 0.0f ? 0.0f : from_bits32((unsigned)(ee + 127) << 23) * ((float)(lo32(e4) & 0x1FFFFFFFu) * 2.220446049250313e-16f)};
      c = side2(s, e, X3, ep, a.minb < 7.0368744e13f * eps);  // 2^46 eps
      ret |= 5 << side;
    }
    const double u = unfix(lin + corr_int(c), E);
    if (side)
      ur = u;
    else
      ul = u;
  }
  return (ret & 3) | (ret & 12 ? 4 : 0);
}

}  // namespace isw
}  // namespace wcns
