// fcs_div.cuh -- division by a number whose reciprocal is at hand.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define FCS_HD __host__ __device__ __forceinline__
#else
#define FCS_HD inline
#endif

namespace fcs {

// x / g from inv = 1 / g, g > 0: the product and one residual correction
// (P. Markstein, Computation of elementary functions on the IBM RISC
// System/6000 processor, IBM J. Res. Dev. 34, 1990), within one unit in the
// last place where no step underflows.  Where x, g or the product is infinite
// the residual is not finite and so the result is NaN; with INF that is looked
// for, and the product, which is the quotient then, returned.  A division
// would cost the solves that use it their registers (its slow path is a call).
template <bool INF>
FCS_HD float quotient(float x, float g, float inv) {
  const float q = x * inv;
  const float r = fmaf(-q, g, x);
  if (INF && !(fabsf(r) <= 3.402823466e38f)) return q;
  return fmaf(r, inv, q);
}

}  // namespace fcs
