// Square root and its inverse from an estimate.
#pragma once

#ifndef __CUDACC__
#include <cmath>
#endif

namespace krr {

// d = sqrt(p) and r = 1 / d from y = (1 + t) / sqrt(p), |t| <= 2^-21: with e = 1 - p
// y^2, 1 / sqrt(p) = y (1 - e)^(-1/2), of whose binomial series the terms to e^2
// are kept (Householder's method of order two for y^-2 = p; A. S. Householder, The
// Numerical Treatment of a Single Nonlinear Equation, 1970), the next one, 5/16
// e^3, being below 2^-61; then one step of Heron's iteration for d, q + (p - q^2)
// / (2 q), with the residual exact by a fused multiply-add and 1 / q = r.  d is
// within 0.51 units of the last place of the root, r within 2^-52.4 of the inverse.
#ifdef __CUDACC__
__host__ __device__ __forceinline__
#else
inline
#endif
void sqrt_from_estimate(double p, double y, double *d, double *r) {
  const double t = p * y;
  const double e = fma(-t, y, 1.0);
  const double y1 = fma(y * e, fma(e, 0.375, 0.5), y);
  const double q = p * y1;
  *d = fma(fma(-q, q, p), 0.5 * y1, q);
  *r = y1;
}

}  // namespace krr
