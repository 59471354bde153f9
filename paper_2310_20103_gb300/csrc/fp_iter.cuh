// Reciprocals and roots from the hardware's approximations: the iterations of
// the kernels whose serial chains or FP64 rate full divisions and square roots
// would set.  Each is tested against CUDA's own operations
// (tests/test_gpu_fp_iter.py).
#pragma once

#include <cuda_runtime.h>

namespace lgw {

// 1/d for a positive d: the hardware's estimate (relative error 2^-20) and one
// step of Householder's iteration of third order for 1/y - d (A. S. Householder,
// The Numerical Treatment of a Single Nonlinear Equation, 1970), y (1 + e + e^2)
// with e = 1 - d y: error 2^-60 before the last rounding, so within one unit of
// the rounded quotient.  3 FP64 operations where the division takes about 10.
// Exponents where the estimate could leave the normal range divide.
__device__ __forceinline__ double pole_rcp(double d) {
  if ((unsigned)(__double2hiint(d) - (32 << 20)) >= (unsigned)(1980 << 20)) return 1.0 / d;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  double e = fma(-d, y, 1.0);
  e = fma(e, e, e);
  return fma(y, e, y);
}

// 1 / sqrt(d), 1e-280 < d < 1e280, to about a unit: the hardware's approximation
// (2^-20 or better) and one step of Householder's iteration of third order for
// 1/y^2 - d, y (1 + e/2 + 3 e^2/8) with e = 1 - d y^2.
__device__ __forceinline__ double rsqrt_iter(double d) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d * y, y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// sqrt(d) and x / s, within one unit, from r ~ 1 / s: one Newton correction with
// the residual of a fused multiply-add (P. W. Markstein, IBM J. Res. Dev. 34
// (1990) 111), instead of a square root and a division (a serial chain of tens
// of FP64 operations) per column.
__device__ __forceinline__ double sqrt_from(double d, double r) {
  const double s = d * r;
  return fma(fma(-s, s, d), 0.5 * r, s);
}
__device__ __forceinline__ double div_from(double x, double s, double r) {
  const double q = x * r;
  return fma(fma(-q, s, x), r, q);
}

}  // namespace lgw
