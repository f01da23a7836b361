// Reciprocals and the scalars of a Householder reflector with few dependent FP64
// instructions: the hardware's estimate (rcp.approx / rsqrt.approx, relative error
// about 2^-23) and one step of third order.
#pragma once

#include <cuda_runtime.h>

namespace ltgw {

// 1/q: with e = 1 - q y, y (1 + e + e^2), the hyperpower iteration of order three
// (M. Altman, Pacific J. Math. 10 (1960) 1107).  e^3 is 2^-69: what is left is the
// rounding of the last operation, 1.01 u (u = 2^-53).  |q| within the normal range.
__device__ __forceinline__ double recip_cubic(double q) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(q));
  const double e = fma(-q, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// tau, beta and sc of the reflector that maps (alpha, x') to (beta, 0), |x'|^2 =
// sigma.  One thread's FP64 instructions follow one another at 64 clocks, comparisons
// included, so: 1/sqrt(s) as y (1 + e/2 + 3 e^2/8), e = 1 - s y^2 (the first terms of
// the binomial series of (1 - e)^(-1/2)), signs and ranges on the integer pipe; 12
// instructions instead of about 28 with Newton steps and FP64 comparisons, and
// 2700 clocks of the fused kernel's step with the IEEE square root and divisions.
// Errors beside the rounding of s: e has that of s y, u, so 1/sqrt(s) 1.6 u and
// sqrt(s) 2.6 u; tau 2.6 u, beta 2.6 u, sc 4.7 u (IEEE operations: 3, 1 and 3).
// Outside the range where the squares are safe, IEEE operations.
__device__ __forceinline__ void reflector_scalars(double alpha, double sigma, double *tau, double *beta, double *sc) {
  if (((__double2hiint(sigma) & 0x7fffffff) | __double2loint(sigma)) == 0) { *tau = 0.0; *beta = alpha; *sc = 0.0; return; }
  const double s = fma(alpha, alpha, sigma), aa = fabs(alpha);
  const int ex = __double2hiint(s) >> 20;   // biased exponent; above 2047: the sign
  double nrm, rinv, rden;
  if ((unsigned)(ex - 223) < 1600u) {       // 2^-800 <= s < 2^800
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
    const double e = fma(-s * y, y, 1.0);
    rinv = fma(y * e, fma(e, 0.375, 0.5), y);
    nrm = s * rinv;
    rden = recip_cubic(aa + nrm);
  } else {
    nrm = sqrt(s);
    rinv = 1.0 / nrm;
    rden = 1.0 / (aa + nrm);
  }
  const bool neg = __double2hiint(alpha) < 0;
  *beta = neg ? nrm : -nrm;
  *tau = fma(aa, rinv, 1.0);                            // (beta - alpha) / beta
  *sc = neg ? -rden : rden;                             // 1 / (alpha - beta)
}

}  // namespace ltgw
