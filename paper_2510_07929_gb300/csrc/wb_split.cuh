// Splitting of L^{-1} r for the double-float Woodbury apply (precond.cu; the CG step kernel of
// solver.cu does it on the fly).
#pragma once
#include "kqr_internal.h"

namespace kqr {

__device__ __forceinline__ void df_split(double x, float& hi, float& lo) {
  hi = (float)x;
  lo = (float)(x - (double)hi);
}
// e with 2^e about sqrt(rr) (rr = ||r||^2), or about rr (is_max: rr = max |r|).
__device__ __forceinline__ int norm_exponent(double rr, bool is_max) {
  const int ex = (int)((__double_as_longlong(rr) >> 52) & 0x7ff) - 1023;
  return is_max ? max(-1000, min(1000, ex)) : ex >> 1;
}
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
__device__ __forceinline__ int max_exponent(unsigned long long wmax) {   // of max L^{-1}; 0 if it is not a normal number
  const int ex = (int)((wmax >> 52) & 0x7ff);
  return ex > 0 && ex < 2046 ? ex - 1023 : 0;
}

}  // namespace kqr
