// usp_dual.cuh -- forward-mode derivative numbers for the gradient form of the
// particle update: a value and its derivatives with respect to three
// parameters (Z_rot, the viscosity index omega, the wall temperature).
//
// Every arithmetic operation and elementary function below propagates the
// derivative by the chain rule; comparisons look at the value only, so a
// discrete decision (a level jump, a cell index, a wall hit, a branch) taken
// in the derivative form is the same as in the plain form of the same
// precision and is held fixed in the derivative (the pathwise derivative
// under common random numbers).
//
// Dual<double> (D3) carries FP64 values and derivatives (the FP64 gradient
// form); Dual<float> (F3) carries FP32 values and derivatives for the
// per-particle arithmetic of the FP32 gradient form, whose cell sums and
// cell-level quantities stay D3 (FP64 accumulation).
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "usp_device.cuh"

namespace usp {
namespace dual {

constexpr int kND = 3;

// elementary functions of the value type: FP32 the library's, FP64 those of
// usp_math.cuh (a derivative number's division took four divisions by the
// same value, 38 FP64 operations of a particle's lane; now 23)
__device__ inline float vsqrt(float x) { return sqrtf(x); }
__device__ inline double vsqrt(double x) { return sqrt_fast(x); }
__device__ inline float vlog(float x) { return logf(x); }
__device__ inline double vlog(double x) { return d_log(x); }
__device__ inline float vexp(float x) { return expf(x); }
__device__ inline double vexp(double x) { return ::exp(x); }
// exp(x) - 1 and its derivative
__device__ inline float vexpm1(float x, float& df) { df = expf(x); return expm1f(x); }
__device__ inline double vexpm1(double x, double& df) {
  const double e = ::expm1(x);
  df = e + 1.0;
  return e;
}
__device__ inline float vcos(float x) { return cosf(x); }
__device__ inline double vcos(double x) { return ::cos(x); }
__device__ inline float vsin(float x) { return sinf(x); }
__device__ inline double vsin(double x) { return ::sin(x); }
__device__ inline float vacos(float x) { return acosf(x); }
__device__ inline double vacos(double x) { return ::acos(x); }
__device__ inline float vcbrt(float x) { return cbrtf(x); }
__device__ inline double vcbrt(double x) { return ::cbrt(x); }
// a / b, and the same for y = 1 / b known (FP64: the value's and the derivatives'
// quotients share it)
__device__ inline float vdiv(float a, float b) { return a / b; }
__device__ inline double vdiv(double a, double b) { return d_div(a, b); }
__device__ inline float vrcp(float) { return 0.0f; }
__device__ inline double vrcp(double b) { return d_rcp(b); }
__device__ inline float vdiv_by(float a, float b, float) { return a / b; }
__device__ inline double vdiv_by(double a, double b, double y) { return d_div_by(a, b, y); }

template <typename V, int N = kND>
struct Dual {
  V v;
  V d[N];
  __host__ __device__ Dual() : v(V(0)) { for (int i = 0; i < N; ++i) d[i] = V(0); }
  __host__ __device__ Dual(double x) : v(V(x)) { for (int i = 0; i < N; ++i) d[i] = V(0); }
  __host__ __device__ Dual(double x, double d0, double d1, double d2) : v(V(x)) {
    d[0] = V(d0); d[1] = V(d1); d[2] = V(d2);
  }
  // between precisions (FP32 particle values <-> FP64 cell values)
  template <typename U>
  __host__ __device__ explicit Dual(const Dual<U, N>& o) : v(V(o.v)) {
    for (int i = 0; i < N; ++i) d[i] = V(o.d[i]);
  }
  __host__ __device__ explicit operator double() const { return (double)v; }
  __host__ __device__ explicit operator float() const { return (float)v; }
  __host__ __device__ explicit operator int() const { return (int)v; }
  __host__ __device__ Dual& operator+=(const Dual& b) {
    v += b.v;
    for (int i = 0; i < N; ++i) d[i] += b.d[i];
    return *this;
  }
  __host__ __device__ Dual& operator-=(const Dual& b) {
    v -= b.v;
    for (int i = 0; i < N; ++i) d[i] -= b.d[i];
    return *this;
  }
  __host__ __device__ Dual& operator*=(const Dual& b) {
    for (int i = 0; i < N; ++i) d[i] = d[i] * b.v + v * b.d[i];
    v *= b.v;
    return *this;
  }
  // y = 1 / b.v
  __device__ Dual& div_by(const Dual& b, V y) {
    const V q = vdiv_by(v, b.v, y);
    for (int i = 0; i < N; ++i) d[i] = vdiv_by(d[i] - q * b.d[i], b.v, y);
    v = q;
    return *this;
  }
  __device__ Dual& operator/=(const Dual& b) {
    return div_by(b, vrcp(b.v));
  }
};

using D3 = Dual<double>;
using F3 = Dual<float>;

// A cell's chains of FP64 operations run on one thread, and a warp's FP64
// instruction takes 64 cycles whatever the number of its lanes that work.  In the
// derivative form lane i of three carries the value and derivative i: three
// operations for a product in place of seven.  Lanes<S>::type is that number
// (S itself in the plain forms, one lane), lane_part and put_part convert.
template <typename S>
struct Lanes {
  using type = S;
  static constexpr int n = 1;
};
template <>
struct Lanes<D3> {
  using type = Dual<double, 1>;
  static constexpr int n = kND;
};
__device__ inline double lane_part(double x, int) { return x; }
__device__ inline Dual<double, 1> lane_part(const D3& x, int i) {
  Dual<double, 1> r(x.v);
  r.d[0] = x.d[i];
  return r;
}
__device__ inline void put_part(double& x, double y, int) { x = y; }
__device__ inline void put_part(D3& x, const Dual<double, 1>& y, int i) {
  if (i == 0) x.v = y.v;
  x.d[i] = y.d[0];
}

template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator+(Dual<V, N> a, const Dual<V, N>& b) { return a += b; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator-(Dual<V, N> a, const Dual<V, N>& b) { return a -= b; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator*(Dual<V, N> a, const Dual<V, N>& b) { return a *= b; }
template <typename V, int N>
__device__ inline Dual<V, N> operator/(Dual<V, N> a, const Dual<V, N>& b) { return a /= b; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator+(Dual<V, N> a, double b) { a.v += V(b); return a; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator+(double b, Dual<V, N> a) { a.v += V(b); return a; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator-(Dual<V, N> a, double b) { a.v -= V(b); return a; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator-(double b, const Dual<V, N>& a) {
  Dual<V, N> r;
  r.v = V(b) - a.v;
  for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
  return r;
}
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator*(Dual<V, N> a, double b) {
  const V c = V(b);
  a.v *= c;
  for (int i = 0; i < N; ++i) a.d[i] *= c;
  return a;
}
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator*(double b, Dual<V, N> a) { return a * b; }
template <typename V, int N>
__device__ inline Dual<V, N> operator/(Dual<V, N> a, double b) {
  const V c = V(b), y = vrcp(c);
  a.v = vdiv_by(a.v, c, y);
  for (int i = 0; i < N; ++i) a.d[i] = vdiv_by(a.d[i], c, y);
  return a;
}
template <typename V, int N>
__device__ inline Dual<V, N> operator/(double b, const Dual<V, N>& a) { return Dual<V, N>(b) / a; }
template <typename V, int N>
__host__ __device__ inline Dual<V, N> operator-(const Dual<V, N>& a) {
  Dual<V, N> r;
  r.v = -a.v;
  for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
  return r;
}

#define USP_DUAL_CMP(op)                                                                       \
  template <typename V, int N>                                                                 \
  __host__ __device__ inline bool operator op(const Dual<V, N>& a, const Dual<V, N>& b) {      \
    return a.v op b.v;                                                                         \
  }                                                                                            \
  template <typename V, int N>                                                                 \
  __host__ __device__ inline bool operator op(const Dual<V, N>& a, double b) { return a.v op b; } \
  template <typename V, int N>                                                                 \
  __host__ __device__ inline bool operator op(double a, const Dual<V, N>& b) { return a op b.v; }
USP_DUAL_CMP(<)
USP_DUAL_CMP(>)
USP_DUAL_CMP(<=)
USP_DUAL_CMP(>=)
USP_DUAL_CMP(==)
USP_DUAL_CMP(!=)
#undef USP_DUAL_CMP

// f(a) with f'(a) = df
template <typename V, int N>
__host__ __device__ inline Dual<V, N> chain(const Dual<V, N>& a, V fv, V df) {
  Dual<V, N> r;
  r.v = fv;
  for (int i = 0; i < N; ++i) r.d[i] = df * a.d[i];
  return r;
}

template <typename V, int N>
__device__ inline Dual<V, N> sqrt(const Dual<V, N>& a) {
  const V s = vsqrt(a.v);
  return chain(a, s, s > V(0) ? vdiv(V(0.5), s) : V(0));
}
// f + a b (FP32: the value by one fused operation whatever is compiled around it, so
// that the form's values do not depend on it)
__device__ inline Dual<float> madd(const Dual<float>& f, const Dual<float>& a,
                                   const Dual<float>& b) {
  Dual<float> r;
  r.v = __fmaf_rn(a.v, b.v, f.v);
  for (int i = 0; i < kND; ++i) r.d[i] = f.d[i] + (a.d[i] * b.v + a.v * b.d[i]);
  return r;
}
template <int N>
__device__ inline Dual<double, N> madd(const Dual<double, N>& f, const Dual<double, N>& a,
                                       const Dual<double, N>& b) {
  Dual<double, N> r;
  r.v = fma(a.v, b.v, f.v);
  for (int i = 0; i < N; ++i) r.d[i] = fma(a.d[i], b.v, fma(a.v, b.d[i], f.d[i]));
  return r;
}
template <typename V, int N>
__device__ inline Dual<V, N> log(const Dual<V, N>& a) { return chain(a, vlog(a.v), vdiv(V(1), a.v)); }
template <typename V, int N>
__device__ inline Dual<V, N> exp(const Dual<V, N>& a) {
  const V e = vexp(a.v);
  return chain(a, e, e);
}
template <typename V, int N>
__device__ inline Dual<V, N> expm1(const Dual<V, N>& a) {
  V df;
  const V e = vexpm1(a.v, df);
  return chain(a, e, df);
}
template <typename V, int N>
__device__ inline Dual<V, N> cos(const Dual<V, N>& a) { return chain(a, vcos(a.v), -vsin(a.v)); }
template <typename V, int N>
__device__ inline Dual<V, N> acos(const Dual<V, N>& a) {
  const V den = vsqrt(V(1) - a.v * a.v);
  return chain(a, vacos(a.v), den > V(0) ? V(-1) / den : V(0));
}
template <typename V, int N>
__device__ inline Dual<V, N> cbrt(const Dual<V, N>& a) {
  const V c = vcbrt(a.v);
  return chain(a, c, c != V(0) ? vdiv(c, V(3) * a.v) : V(0));
}
template <typename V, int N>
__device__ inline Dual<V, N> fabs(const Dual<V, N>& a) { return a.v < V(0) ? -a : a; }
template <typename V, int N>
__device__ inline Dual<V, N> fmin(const Dual<V, N>& a, const Dual<V, N>& b) { return b.v < a.v ? b : a; }
template <typename V, int N>
__device__ inline Dual<V, N> fmax(const Dual<V, N>& a, const Dual<V, N>& b) { return b.v > a.v ? b : a; }
template <typename V, int N>
__device__ inline V value(const Dual<V, N>& a) { return a.v; }

}  // namespace dual

using dual::D3;
using dual::F3;
using dual::kND;
using dual::value;
__device__ inline double value(double a) { return a; }
__device__ inline float value(float a) { return a; }

// A quantity held at its value in the gradient form: its derivative is
// dropped (the identity in the plain forms).
template <typename V, int N>
__device__ inline dual::Dual<V, N> held(const dual::Dual<V, N>& a) { return dual::Dual<V, N>(a.v); }
__device__ inline double held(double a) { return a; }
__device__ inline float held(float a) { return a; }

}  // namespace usp
