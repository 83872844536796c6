// Scalar FP64 helpers for code in which the latency of a chain of FP64 instructions counts: a
// warp-wide FP64 instruction holds its sub-partition's pipe for 64 clocks on GB300, however few
// lanes are active.
#pragma once
#include <cuda_runtime.h>

namespace tdmrg {

// biased exponent of a double (2047: Inf or NaN)
__device__ __forceinline__ int bexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// 1 / sqrt(x) for a positive normal x: single-precision seed y, then the series of
// (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + ... for e = 1 - x y^2 (|e| < 2^-20, so the next term is below
// 2^-61).  Five FP64 instructions: a warp-wide one holds its pipe for 64 clocks here.
__device__ __forceinline__ double rsqrt_series(double x) {
  const long long b = __double_as_longlong(x);
  const int k = ((int)(b >> 52) - 1023) >> 1;                  // x = xs 4^k, xs in [1, 4)
  const double xs = __longlong_as_double(b - (long long)(2 * k) * (1LL << 52));
  const double y0 = (double)rsqrtf(__double2float_rn(xs));
  const double t = xs * y0;
  const double e = fma(-t, y0, 1.0);
  const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);
  return __longlong_as_double(__double_as_longlong(y) - (long long)k * (1LL << 52));
}

}  // namespace tdmrg
