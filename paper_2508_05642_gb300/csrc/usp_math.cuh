// usp_math.cuh -- FP64 elementary functions for the per-cell closed forms and
// the FP64 particle arithmetic, written for few FP64 operations.  Each quarter
// of an SM has half an FP64 lane per clock: a warp's FP64 instruction occupies
// it for 64 cycles, however many lanes are active and whether or not the next
// one depends on it, so the time of a cell's coefficients is their count.  Against
// timed loops of multiply-adds the library's division, square root and logarithm take
// 10, 10 and 35 such slots; those below 7, 6 and 28.  (CUDA's exp, expm1 and cbrt, 17, 21
// and 18, are used as they are: forms as exact as theirs saved nothing.)
// Every function answers every argument: those outside the range stated at it
// (zero, denormal, negative, very large, infinite, not a number) take CUDA's
// own function, in a call of its own so that its code is not at every use.
#pragma once

#include <cuda_runtime.h>

namespace usp {

constexpr double kLn2Hi = 0x1.62e42fefa2p-1;        // 40 bits: times an exponent exact
constexpr double kLn2Lo = 0x1.9ef35793c7673p-41;    // ln 2 - kLn2Hi

// zero, denormal, infinite or not a number (integer work, beside the FP64 pipe)
__device__ __forceinline__ bool d_ends(double b) {
  return ((unsigned)__double2hiint(b) & 0x7ff00000u) - 0x00100000u >= 0x7fe00000u;
}
__device__ __forceinline__ bool d_zero(double a) {
  return ((__double2hiint(a) & 0x7fffffff) | __double2loint(a)) == 0;
}
// x > 0 and x < 0 by the bits: a comparison occupies the FP64 pipe like a product
__device__ __forceinline__ bool d_pos(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool d_neg(double x) { return d_pos(-x); }
static __device__ __noinline__ double d_div_ends(double a, double b) { return a / b; }
static __device__ __noinline__ double d_log_ends(double x) { return log(x); }
static __device__ __noinline__ double d_log1p_inv_ends(double b) { return log1p(1.0 / b); }
static __device__ __noinline__ double d_sqrt_ends(double x) { return sqrt(x); }

// 1 / b: hardware seed (about 2^-20), then y (1 + e + e^2), e = 1 - b y, whose
// remainder is e^3
__device__ __forceinline__ double d_rcp(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  if (d_ends(b) || d_ends(y)) return d_div_ends(1.0, b);
  const double e = fma(-b, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// a / b for y = 1 / b, with the residual of the quotient added (Markstein): the
// rounded quotient, where a y rounds twice
__device__ __forceinline__ double d_div_by(double a, double b, double y) {
  const double q = a * y;
  if (d_ends(b) || d_ends(q)) return d_zero(a) && !d_ends(b) ? q : d_div_ends(a, b);
  return fma(fma(-b, q, a), y, q);
}
__device__ __forceinline__ double d_div(double a, double b) { return d_div_by(a, b, d_rcp(b)); }
// sqrt(x), exponents within +-900: the hardware reciprocal square root (about
// 2^-20), one Goldschmidt step for the root and its half reciprocal together
// and Markstein's residual correction (P. Markstein, "IA-64 and Elementary
// Functions", 2000), five multiply-adds in all
__device__ __forceinline__ double d_sqrt(double x) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - (123 << 20)) > (unsigned)(1800 << 20)) return d_sqrt_ends(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y;
  double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));   // y / 2
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, x), h, g);
}
// the same with 1 / sqrt(x) in rs: twice the half reciprocal, one more step
__device__ __forceinline__ double d_sqrt(double x, double& rs) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - (123 << 20)) > (unsigned)(1800 << 20)) {
    const double s = d_sqrt_ends(x);
    rs = d_div_ends(1.0, s);
    return s;
  }
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y;
  double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));   // y / 2
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  g = fma(fma(-g, g, x), h, g);
  y = __hiloint2double(__double2hiint(h) + 0x00100000, __double2loint(h));          // 2 h
  rs = fma(y, fma(-g, y, 1.0), y);
  return g;
}

// E ln 2 + 2 atanh f, f = num / (den + rest), |f| <= 0.18, |E ln 2| above |2 f| or 0.  f is
// a quotient q and its rest lo; 2 atanh f = 2 f + f^3 P(f^2), P interpolating (2 atanh
// f - 2 f) / f^3 at the Chebyshev points of f^2 in [0, 0.0297] (error below 2^-57 of
// the result); what the sum E ln 2 + 2 q rounds off goes into the last addition.
__device__ __forceinline__ double d_log_sum(double num, double den, double rest, double E) {
  const double y = d_rcp(den), q = num * y;
  const double lo = fma(-rest, q, fma(-den, q, num)) * y;
  const double z = q * q;
  double p = fma(0x1.2b9f7fb3de73fp-3, z, 0x1.39f8963ccbdc2p-3);
  p = fma(p, z, 0x1.7462e17b4cdd0p-3);
  p = fma(p, z, 0x1.c71c6247410e3p-3);
  p = fma(p, z, 0x1.2492492e6dfddp-2);
  p = fma(p, z, 0x1.9999999994e76p-2);
  p = fma(p, z, 0x1.5555555555558p-1);
  const double t = fma(E, kLn2Lo, fma(q * z, p, 2.0 * lo));
  const double a = fma(E, kLn2Hi, 2.0 * q);
  return a + (t + fma(2.0, q, fma(E, kLn2Hi, -a)));
}
// log x, x above 0 and normal: x = 2^e m, m in [sqrt 1/2, sqrt 2), f = (m - 1) / (m + 1)
__device__ __forceinline__ double d_log(double x) {
  const int hi = __double2hiint(x);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return d_log_ends(x);
  const int e = (hi - 0x3fe6a09e) >> 20;
  const double m = __hiloint2double(hi - (e << 20), __double2loint(x)), den = m + 1.0;
  return d_log_sum(m - 1.0, den, m - (den - 1.0), (double)e);
}
// log(1 + 1/b), b in [2^-100, 2^100]: with (1 + b) / b = 2^e m, f = (1 + b - 2^e b) / (1 + b
// + 2^e b), so that nothing is lost for large b (e = 0, f = 1 / (2 b + 1)); e from FP32
__device__ __forceinline__ double d_log1p_inv(double b) {
  if ((unsigned)(__double2hiint(b) - (923 << 20)) > (unsigned)(200 << 20)) return d_log1p_inv_ends(b);
  const float x = 1.0f + __frcp_rn((float)b);
  int e = (__float_as_int(x) - 0x3f3504f3) >> 23;
  e = e < 0 ? 0 : e;
  const double s = __hiloint2double((e + 1023) << 20, 0);   // 2^e
  const double c = 1.0 + s, den = fma(b, c, 1.0);
  // what the denominator rounds off, its larger part taken away first
  const double rest = b > 1.0 ? fma(b, c, -den) + 1.0 : fma(b, c, 1.0 - den);
  return d_log_sum(fma(b, 1.0 - s, 1.0), den, rest, (double)e);
}

}  // namespace usp
