// Packed FP32 arithmetic: an f2 holds one value at two grid points, and every
// operation is one instruction on both (add / mul / fma.rn.f32x2 of sm_100 and
// later).  Each half rounds exactly like the scalar operation.
//
// On GB300 a packed instruction runs at the FMA pipe's lane rate (measured 117
// lanes per clock and SM for FADD2 and FMUL2, 106 for FFMA2, like their scalar
// forms) but takes one issue slot for two lanes.  Subtraction is the fma with
// -1 (exact product, one rounding): there is no packed negation.
#pragma once

#include <cuda_runtime.h>

namespace snk {

// the f2 overload of fma below must not hide the FP64 / FP32 ones
using ::fma;

struct f2 {
  float2 v;
  f2() = default;
  __device__ __forceinline__ f2(float x, float y) : v(make_float2(x, y)) {}
  __device__ __forceinline__ explicit f2(float x) : v(make_float2(x, x)) {}
  __device__ __forceinline__ explicit f2(int x) : v(make_float2((float)x, (float)x)) {}
  __device__ __forceinline__ explicit f2(float2 x) : v(x) {}
};

__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return f2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator-(f2 a) { return f2(-a.v.x, -a.v.y); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return fma(b, f2(-1.0f), a); }
__device__ __forceinline__ f2& operator+=(f2& a, f2 b) {
  a = a + b;
  return a;
}

}  // namespace snk
