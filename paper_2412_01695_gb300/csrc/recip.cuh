// 1 / x and 1 / sqrt(x) for the serial parts of the reduced eigensolver, by the Newton-Raphson
// iterations r += r (1 - x r) and r += r (1 - x r^2) / 2 from the hardware's approximation (about
// 20 correct bits; two steps give 53).  The last step's correction is added with one rounding, and
// the residual of 1 / x is exact, so fast_rcp is within 0.501 units in the last place, as close as
// the division; in fast_rsqrt the product x r / 2 is rounded once more: within 1.01 units,
// where 1.0 / sqrt(x) with its two roundings is within 1.5 (largest found over the ranges below:
// 0.500, 0.987 and 1.470; the division 0.500).
//
// Ranges: |x| in [1e-290, 1e290] for fast_rcp, x in [1e-280, 1e280] for fast_rsqrt.  Outside the
// approximation flushes to zero or infinity and the steps give NaN; callers keep their pivots
// inside (Sturm pivots at least 1e-290 max(1, e^2), which bounds the next one by 1e290; LDL^T
// pivots above 2e-16) or fall back to the division.
#pragma once
#include <cuda_runtime.h>

namespace pwk {

__device__ __forceinline__ double fast_rcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(fma(-x, r, 1.0), r, r);
  return fma(fma(-x, r, 1.0), r, r);
}
__device__ __forceinline__ double fast_rsqrt(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double h = 0.5 * x;
  r = fma(fma(-h * r, r, 0.5), r, r);
  return fma(fma(-h * r, r, 0.5), r, r);
}

}  // namespace pwk
