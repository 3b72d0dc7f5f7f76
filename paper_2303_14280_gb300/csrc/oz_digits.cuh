// Signed base-2^8 digits of a fixed-point remainder, for the slicing of the split
// products (kernels_ozaki.cu).  Plain integer arithmetic that any C++ compiler
// takes, so that it can be checked on the host.
#pragma once

#ifdef __CUDACC__
#define SNK_DIGIT_FN __host__ __device__ __forceinline__
#else
#define SNK_DIGIT_FN inline
#endif

namespace snk {

// Takes the next digit off r at bit k > 0: the nearest integer to r 2^-k, ties up;
// r becomes what is left, in [-2^(k-1), 2^(k-1)).  Any r is allowed at k = 24, |r|
// <= 2^30 below.  d = 128 at k = 24 (r >= 2^31 - 2^23) makes d 2^k = 2^31, which an
// int does not hold, so the remainder is formed in unsigned arithmetic.
SNK_DIGIT_FN int oz_take_digit(int& r, int k) {
  const int d = k == 24 ? (r >> 24) + ((r >> 23) & 1) : (r + (1 << (k - 1))) >> k;
  r = (int)((unsigned)r - ((unsigned)d << k));
  return d;
}

}  // namespace snk
