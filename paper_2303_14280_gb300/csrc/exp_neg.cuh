// e^{-x} for 0 <= x < 700 in FP64 with nine FP64 operations, by the table-driven
// method (P. T. P. Tang, ACM Trans. Math. Softw. 15, 144, 1989): x = k ln2/256 +
// r with |r| <= ln2/512, e^{-x} = 2^{-k/256} e^{-r}; 2^{-j/256}, j < 256, comes from a
// table in shared memory as the double T and its relative error t, the remaining
// power of two goes into the exponent bits, and e^{-r} - 1 is its Taylor polynomial
// of degree 4 (the next term is below 4e-17), to which t is added by the multiply-add
// that would be its last multiplication.  ln2/256 is split into a 32-bit head, so that
// k head is exact, and a tail.  Relative error at most 1.5e-16: the last rounding and
// the polynomial's truncation (2.4e-16 without t).
//
// FP64 issues at 2 lanes per clock and SM on GB300, so the number of FP64
// operations is what the collocation kernels cost.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "snk_internal.h"

namespace snk {

// 2^{-j/256} = tab[j].x (1 + tab[j].y)
inline void exp_table_fill(double2* tab) {
  for (int j = 0; j < kExpTable; ++j) {
    const long double v = exp2l(-(long double)j / kExpTable);
    tab[j].x = (double)v;
    tab[j].y = (double)((v - (long double)tab[j].x) / v);
  }
}

__device__ __forceinline__ void exp_table_load(double2* tab, const double2* __restrict__ gtab) {
  for (int e = threadIdx.x; e < kExpTable; e += blockDim.x) tab[e] = gtab[e];
  __syncthreads();
}

__device__ __forceinline__ double exp_neg(double x, const double2* tab) {
  constexpr double kMagic = 0x1.8p52;  // adding it rounds to an integer in the low word
  const double t = fma(x, 0x1.71547652b82fep+8, kMagic);  // 256 / ln2
  const int k = __double2loint(t);
  const double kd = t - kMagic;
  double r = fma(-kd, 0x1.62e42fee00000p-9, x);
  r = fma(-kd, 0x1.a39ef35793c76p-41, r);
  double q = fma(r, 1.0 / 24.0, -1.0 / 6.0);
  q = fma(q, r, 0.5);
  q = fma(q, r, -1.0);
  const double2 T = tab[k & (kExpTable - 1)];
  const double e = fma(T.x, fma(q, r, T.y), T.x);
  return __hiloint2double(__double2hiint(e) - ((k >> 8) << 20), __double2loint(e));
}

// e^{-a_k r^2} of a shell's primitives for k < n <= kRadialPrims into e, zero
// beyond the cut.
__device__ __forceinline__ void radial_exps(const double* __restrict__ exps, int n, double r2, double cut,
                                            const double2* tab, double (&e)[kRadialPrims]) {
#pragma unroll
  for (int k = 0; k < kRadialPrims; ++k) {
    e[k] = 0.0;
    if (k < n) {
      const double x = exps[k] * r2;
      if (x < cut) e[k] = exp_neg(x, tab);
    }
  }
}

}  // namespace snk
