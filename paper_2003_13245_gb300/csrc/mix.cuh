// One entry of a sparse MPO mixing, shared by the kernel that stores the mixed tensor and by the
// digit split that mixes on the fly.
#pragma once
#include "tdmrg_internal.cuh"

namespace tdmrg {

// acc += v z (`first`: acc is zero)
__device__ __forceinline__ void mix_add(cplx& acc, cplx v, cplx z, bool first) {
  // (entries of 1 and real entries are told apart by their bits: comparisons run at the FP64 rate)
  if (__double_as_longlong(v.y) == 0) {
    if (first && __double_as_longlong(v.x) == 0x3ff0000000000000LL) {
      acc = z;
    } else {
      acc.x = fma(v.x, z.x, acc.x);
      acc.y = fma(v.x, z.y, acc.y);
    }
  } else {
    acc.x = fma(v.x, z.x, fma(-v.y, z.y, acc.x));
    acc.y = fma(v.x, z.y, fma(v.y, z.x, acc.y));
  }
}

// sum over the entries [lo, hi) of val * x[chan * xs + u * dmb], in order
__device__ __forceinline__ cplx mix_entries(int lo, int hi, const int2* cu, const cplx* val,
                                            const cplx* x, long long xs, int dmb) {
  cplx acc = make_double2(0.0, 0.0);
  for (int e = lo; e < hi; ++e) {
    const int2 c = __ldg(cu + e);
    mix_add(acc, __ldg(val + e), x[c.x * xs + (long long)c.y * dmb], e == lo);
  }
  return acc;
}

}  // namespace tdmrg
