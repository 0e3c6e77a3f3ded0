// usp_math.cuh -- FP64 elementary functions for the per-cell closed forms and
// the FP64 particle arithmetic, written for few FP64 operations.  Each quarter
// of an SM has half an FP64 lane per clock: a warp's FP64 instruction occupies
// it for 64 cycles, however many lanes are active and whether or not the next
// one depends on it, so the time of a cell's coefficients is their count.  The
// library's division, square root, logarithm, exponential, expm1 and cbrt take
// 10, 11, 32, 17, 21 and 18 such slots with the branches for special
// arguments; those below 8, 9, 20, 16, 17 and 16 without a branch.  They hold for
// normal positive arguments (division: normal denominators of either sign)
// with errors of at most one unit in the last place; zero, infinite and NaN
// arguments give infinities or NaN.
#pragma once

#include <cuda_runtime.h>

namespace usp {

constexpr double kLn2Hi = 0x1.62e42fefa2p-1;        // 40 bits: times an exponent exact
constexpr double kLn2Lo = 0x1.9ef35793c7673p-41;    // ln 2 - kLn2Hi
constexpr double kLog2e = 0x1.71547652b82fep+0;

// zero, denormal, infinite or not a number (integer work, beside the FP64 pipe)
__device__ __forceinline__ bool d_ends(double b) {
  return ((unsigned)__double2hiint(b) & 0x7ff00000u) - 0x00100000u >= 0x7fe00000u;
}
// 1 / b: hardware seed (about 2^-20), then y (1 + e + e^2), e = 1 - b y, whose
// remainder is e^3; the seed itself where b has no such e (0 of an infinity, an
// infinity of 0)
__device__ __forceinline__ double d_rcp(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  const double e = fma(-b, y, 1.0);
  return d_ends(b) ? y : fma(y, fma(e, e, e), y);
}
// a / b with the residual of the quotient added (Markstein)
__device__ __forceinline__ double d_div(double a, double b) {
  const double y = d_rcp(b), q = a * y;
  return d_ends(b) || d_ends(a) ? q : fma(fma(-b, q, a), y, q);
}
// 1 / sqrt(x): the seed times (1 - e)^(-1/2) to second order, e = 1 - x y^2
__device__ __forceinline__ double d_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
// sqrt(x), x > 0: Goldschmidt's step and Markstein's residual correction
__device__ __forceinline__ double d_sqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, x), h, g);
}

// log((1 + f) / (1 - f)) + E ln 2 for f = q + lo, |f| <= 0.18: 2 f + f^3 P(f^2), P
// interpolating (2 atanh f - 2 f) / f^3 at the Chebyshev points of f^2 in [0, 0.0297]
// (error below 2^-57 of the result)
__device__ __forceinline__ double d_log_sum(double q, double lo, double E) {
  const double z = q * q;
  double p = fma(0x1.2b9f7fb3de73fp-3, z, 0x1.39f8963ccbdc2p-3);
  p = fma(p, z, 0x1.7462e17b4cdd0p-3);
  p = fma(p, z, 0x1.c71c6247410e3p-3);
  p = fma(p, z, 0x1.2492492e6dfddp-2);
  p = fma(p, z, 0x1.9999999994e76p-2);
  p = fma(p, z, 0x1.5555555555558p-1);
  const double t = fma(E, kLn2Lo, fma(q * z, p, 2.0 * lo));
  return fma(E, kLn2Hi, fma(2.0, q, t));
}
// num / den as a quotient and the rest
__device__ __forceinline__ void d_quot(double num, double den, double& q, double& lo) {
  const double y = d_rcp(den);
  q = num * y;
  lo = fma(-den, q, num) * y;
}
// log x, x = 2^e m, m in [sqrt 1/2, sqrt 2): f = (m - 1) / (m + 1)
__device__ __forceinline__ double d_log(double x) {
  const int hi = __double2hiint(x), e = (hi - 0x3fe6a09e) >> 20;
  const double m = __hiloint2double(hi - (e << 20), __double2loint(x));
  double q, lo;
  d_quot(m - 1.0, m + 1.0, q, lo);
  return d_log_sum(q, lo, (double)e);
}
// log(1 + 1/b), b > 0: with (1 + b) / b = 2^e m, f = (1 + b - 2^e b) / (1 + b + 2^e b),
// so that nothing is lost for large b (e = 0, f = 1 / (2 b + 1)); e from FP32
__device__ __forceinline__ double d_log1p_inv(double b) {
  const float x = 1.0f + __frcp_rn((float)b);
  int e = (__float_as_int(x) - 0x3f3504f3) >> 23;
  e = e < 0 ? 0 : e;
  const double s = __hiloint2double((e + 1023) << 20, 0);   // 2^e
  double q, lo;
  d_quot(fma(b, 1.0 - s, 1.0), fma(b, 1.0 + s, 1.0), q, lo);
  return d_log_sum(q, lo, (double)e);
}

// p = exp(r) - 1 and s = 2^k with x = k ln 2 + r, |r| <= ln 2 / 2, for x in
// [-600, 600] (values beyond are taken there): r + r^2 P(r), P interpolating
// (exp(r) - 1 - r) / r^2 at Chebyshev points (error below 2^-59).  exp x = s + s p,
// exp x - 1 = s p + (s - 1).
__device__ __forceinline__ double d_exp_parts(double x, double& s) {
  const int hi = __double2hiint(x);
  if ((hi & 0x7fffffff) > 0x4082c000) x = __hiloint2double((hi & 0x80000000) | 0x4082c000, 0);
  const double t = fma(x, kLog2e, 0x1.8p52);          // k in the low bits
  const int k = __double2loint(t);
  const double K = t - 0x1.8p52;
  const double r = fma(-K, kLn2Lo, fma(-K, kLn2Hi, x));
  double p = fma(0x1.1f7340dbc337ep-29, r, 0x1.af4e554377204p-26);
  p = fma(p, r, 0x1.27e4db46cddd1p-22);
  p = fma(p, r, 0x1.71de01fdbf9cap-19);
  p = fma(p, r, 0x1.a01a01a6e1e2ap-16);
  p = fma(p, r, 0x1.a01a01abf85abp-13);
  p = fma(p, r, 0x1.6c16c16c162c3p-10);
  p = fma(p, r, 0x1.11111111100bep-7);
  p = fma(p, r, 0x1.5555555555556p-5);
  p = fma(p, r, 0x1.5555555555557p-3);
  p = fma(p, r, 0.5);
  s = __hiloint2double((k + 1023) << 20, 0);
  return fma(p * r, r, r);
}
__device__ __forceinline__ double d_expm1(double x) {
  double s;
  const double p = d_exp_parts(x, s);
  return fma(s, p, s - 1.0);
}
__device__ __forceinline__ double d_exp(double x) {
  double s;
  const double p = d_exp_parts(x, s);
  return fma(s, p, s);
}

// the real cube root of a != 0: z = |a|^(-1/3) from FP32, corrected by (1 - r)^(-1/3)
// to third order, r = 1 - |a| z^3; then |a| z^2 and one Newton step
__device__ __forceinline__ double d_cbrt(double a) {
  const double b = fabs(a);
  const float bf = fmaxf((float)b, 1e-30f);
  const double z0 = (double)exp2f(-0.33333334f * log2f(bf));
  const double r = fma(-b, (z0 * z0) * z0, 1.0);
  const double z = fma(z0, r * fma(r, fma(r, 14.0 / 81, 2.0 / 9), 1.0 / 3), z0);
  const double z2 = z * z, y = b * z2;
  const double c = fma(fma(-(y * y), y, b), z2 * (1.0 / 3), y);
  return copysign(c, a);
}

}  // namespace usp
