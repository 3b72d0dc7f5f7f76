// Double-FP32 ("ds") arithmetic: a value is the unevaluated sum hi + lo of two
// floats with |lo| <= ulp(hi) / 2, about 48 significant bits.  Built from the
// error-free transformations of floating-point arithmetic:
//   TwoSum (Knuth):      s + e = a + b exactly, 6 FP32 operations;
//   FastTwoSum (Dekker): the same when |a| >= |b|, 3 operations;
//   TwoProd:             p + e = a b exactly with one FMA, 2 operations.
// Addition adds the low parts into the TwoSum error and renormalises (11
// operations, error ~2^-46 (|x| + |y|)); multiplication keeps the cross terms
// (7 operations, ~2^-46 relative); a fused multiply-add is the product
// followed by the addition (15 operations).  Every step uses the _rn
// intrinsics so that the compiler neither contracts nor reorders them.
//
// On GB300 the FP32 pipe issues 64x the FP64 rate, so ds arithmetic runs
// several times faster than FP64 at a precision (~1e-14 relative) far below
// what the K tolerance needs.
#pragma once

#include <cuda_runtime.h>

namespace snk {

// the ds overload of fma below must not hide the FP64 / FP32 ones
using ::fma;

struct ds {
  float hi, lo;
};

__device__ __forceinline__ ds ds_make(float hi, float lo) {
  ds r;
  r.hi = hi;
  r.lo = lo;
  return r;
}

__device__ __forceinline__ ds ds_from(double v) {
  const float h = __double2float_rn(v);
  return ds_make(h, __double2float_rn(v - (double)h));
}

__device__ __forceinline__ double ds_to(ds a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ ds ds_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return ds_make(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ ds operator+(ds x, ds y) {
  const float s = __fadd_rn(x.hi, y.hi);
  const float bb = __fsub_rn(s, x.hi);
  const float e = __fadd_rn(__fsub_rn(x.hi, __fsub_rn(s, bb)), __fsub_rn(y.hi, bb));
  return ds_fast_two_sum(s, __fadd_rn(e, __fadd_rn(x.lo, y.lo)));
}

__device__ __forceinline__ ds operator-(ds x) { return ds_make(-x.hi, -x.lo); }
__device__ __forceinline__ ds operator-(ds x, ds y) { return x + (-y); }
__device__ __forceinline__ ds& operator+=(ds& x, ds y) {
  x = x + y;
  return x;
}

__device__ __forceinline__ ds operator*(ds x, ds y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return ds_fast_two_sum(p, e);
}

// x times an exactly representable float
__device__ __forceinline__ ds operator*(ds x, float s) {
  const float p = __fmul_rn(x.hi, s);
  float e = __fmaf_rn(x.hi, s, -p);
  e = __fmaf_rn(x.lo, s, e);
  return ds_fast_two_sum(p, e);
}

__device__ __forceinline__ ds fma(ds x, ds y, ds z) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  const float s = __fadd_rn(p, z.hi);
  const float bb = __fsub_rn(s, p);
  const float t = __fadd_rn(__fsub_rn(p, __fsub_rn(s, bb)), __fsub_rn(z.hi, bb));
  return ds_fast_two_sum(s, __fadd_rn(t, __fadd_rn(e, z.lo)));
}

// ---- operations of the generated integral code (os_generated.cuh), for double, float and ds
//
//   dot2(a, b, c, d)           a b + c d
//   dot2_add<m>(a, b, c, d, x) a b + c d + m x, m = 1, 2, 3
//   acc_add / acc_mac          running sums M += x, M += a b;  acc_get reads one
//   acc_lead                   acc_add of a primitive pair's leading scalar; in double
//                              acc_mac by the prefactor, which the FP64 seeds leave out
//
// In ds the products of a dot product stay unnormalised (p + e, 4 operations
// each), the leading parts are added error-free and everything small is
// collected before the one renormalisation: 19 operations for dot2 and 27 for
// dot2_add<1>, against 22 and 33 for the same sum made of fma and operator+,
// with fewer roundings.  A running sum keeps (hi, lo) unnormalised, lo
// collecting the errors (8 operations for acc_add, 12 for acc_mac); a long one is
// renormalised on the way (acc_renorm).

template <class T>
__device__ __forceinline__ T dot2(T a, T b, T c, T d) {
  return fma(a, b, c * d);
}
template <int m, class T>
__device__ __forceinline__ T dot2_add(T a, T b, T c, T d, T x) {
  const T v = fma(a, b, c * d);
  return m == 1 ? v + x : fma(T(m), x, v);
}
template <class T>
__device__ __forceinline__ void acc_add(T& s, T x) {
  s += x;
}
template <class A, class R>
__device__ __forceinline__ void acc_lead(A& s, const R&, const R& x) {
  acc_add(s, x);
}
__device__ __forceinline__ void acc_lead(double& s, double c, double x) { s = ::fma(c, x, s); }
template <class T>
__device__ __forceinline__ void acc_mac(T& s, T a, T b) {
  s = fma(a, b, s);
}
template <class T>
__device__ __forceinline__ T acc_get(T s) {
  return s;
}

// x y = p + e without renormalisation
__device__ __forceinline__ ds ds_mul_raw(ds x, ds y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return ds_make(p, e);
}

// x^2 + y^2 + z^2 as an unnormalised sum (28 operations; 37 with fma)
__device__ __forceinline__ ds ds_sqr_raw(ds x) {
  const float p = __fmul_rn(x.hi, x.hi);
  return ds_make(p, __fmaf_rn(__fadd_rn(x.hi, x.hi), x.lo, __fmaf_rn(x.hi, x.hi, -p)));
}
__device__ __forceinline__ ds ds_two_sum(float a, float b);
__device__ __forceinline__ ds ds_norm2_raw(ds x, ds y, ds z) {
  const ds p = ds_sqr_raw(x), q = ds_sqr_raw(y), r = ds_sqr_raw(z);
  const ds s = ds_two_sum(p.hi, q.hi);
  const ds t = ds_two_sum(s.hi, r.hi);
  return ds_make(t.hi, __fadd_rn(__fadd_rn(t.lo, s.lo), __fadd_rn(__fadd_rn(p.lo, q.lo), r.lo)));
}

// a + b = s + e exactly
__device__ __forceinline__ ds ds_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return ds_make(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

__device__ __forceinline__ ds dot2(ds a, ds b, ds c, ds d) {
  const ds p = ds_mul_raw(a, b), q = ds_mul_raw(c, d);
  const ds s = ds_two_sum(p.hi, q.hi);
  return ds_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(p.lo, q.lo)));
}

template <int m>
__device__ __forceinline__ ds dot2_add(ds a, ds b, ds c, ds d, ds x) {
  if (m == 2) x = ds_make(2.0f * x.hi, 2.0f * x.lo);
  if (m == 3) x = x * 3.0f;
  const ds p = ds_mul_raw(a, b), q = ds_mul_raw(c, d);
  const ds s = ds_two_sum(p.hi, q.hi);
  const ds t = ds_two_sum(s.hi, x.hi);
  return ds_fast_two_sum(t.hi, __fadd_rn(__fadd_rn(t.lo, s.lo), __fadd_rn(__fadd_rn(p.lo, q.lo), x.lo)));
}

__device__ __forceinline__ void acc_add(ds& s, ds x) {
  const ds t = ds_two_sum(s.hi, x.hi);
  s = ds_make(t.hi, __fadd_rn(s.lo, __fadd_rn(t.lo, x.lo)));
}

__device__ __forceinline__ void acc_mac(ds& s, ds a, ds b) {
  const ds p = ds_mul_raw(a, b);
  const ds t = ds_two_sum(s.hi, p.hi);
  s = ds_make(t.hi, __fadd_rn(s.lo, __fadd_rn(t.lo, p.lo)));
}

__device__ __forceinline__ ds acc_get(ds s) { return ds_fast_two_sum(s.hi, s.lo); }

// A running sum brought back to |lo| <= 2^-24 |hi| (3 operations).  Left alone, lo
// grows with the number of terms and its own rounding with it: relative rms error
// of a sum of n terms of one sign, never renormalised / after every term, 1.8e-13 /
// 2.1e-14 at n = 1,000, 3.5e-13 / 3.2e-14 at 2,000, 2.8e-15 / 2.3e-15 at 9.
__device__ __forceinline__ void acc_renorm(ds& s) { s = acc_get(s); }

// 1 / sqrt(t) for t > 0: the FP32 estimate refined by one Newton step in ds
// (the relative error squares: ~1e-14).
__device__ __forceinline__ ds ds_rsqrt(ds t) {
  const float r0 = rsqrtf(t.hi);
  const ds y = (t * r0) * r0;                       // t r0^2 = 1 - d
  const ds h = ds_make(1.0f, 0.0f) - y;              // d
  return ds_make(r0, 0.0f) + (ds_make(r0, 0.0f) * h) * 0.5f;
}

}  // namespace snk
