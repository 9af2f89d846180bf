// 1/d and 1/sqrt(d) in fp64 from the approximate instructions and a power series, for normal d > 0 whose results are normal.
// An approximation x0 leaves a residual; the correction that removes it is an elementary series in it:
//   reciprocal      e0 = 1 - d r0     1/d       = r0 / (1 - e0)       = r0 (1 + e0 + e0^2 + ...)           geometric series
//   its root        f  = 1 - d y0^2   1/sqrt(d) = y0 (1 - f)^(-1/2)   = y0 (1 + f/2 + 3/8 f^2 + ...)       binomial series
// Both stop after the second power. The instructions return 20 bits, so what is cut off is e0^3 < 2^-59 and
// 5/16 f^3 < 2^-58 (f is about twice the relative error of y0); the roundings on the way leave less than 2^-52.
#pragma once

namespace lordo {

// 1/d = r0 (1 + e); the caller multiplies r0 first, which keeps e off its chain
__device__ __forceinline__ void recip_parts(double d, double& r0, double& e) {
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(d));
  const double e0 = fma(-d, r0, 1.0);
  e = fma(e0, e0, e0);
}

__device__ __forceinline__ double recip_sqrt(double d) {
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(d));
  const double f = fma(-d * y0, y0, 1.0);
  return fma(y0, f * fma(3.0 / 8.0, f, 0.5), y0);
}

}  // namespace lordo
