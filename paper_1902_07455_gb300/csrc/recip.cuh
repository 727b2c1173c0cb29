// Reciprocal and reciprocal square root of the eigensolver's and the Cholesky factor's dependent chains.
#pragma once

namespace lrfg {

// 1 / x and 1 / sqrt(x): the hardware's approximation (about 2^-20) improved by one third-order Householder step each
// (error of the order of the cube of the first), about half the latency of a division; outside the approximations'
// range the divisions themselves.  Within one unit in the last place of the exact value for normal results (a division or
// a square root is within half of one).
__device__ __forceinline__ double recip(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  if (ex < 24 || ex > 2022) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = fma(-x, y, 1.0);
  return fma(y, fma(h, h, h), y);
}

__device__ __forceinline__ double recip_sqrt(double x) {
  const int ex = (__double2hiint(x) >> 20) & 0x7ff;
  if (ex < 24 || ex > 2022) return 1.0 / sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = fma(-x * y, y, 1.0);
  return fma(y * h, fma(0.375, h, 0.5), y);
}

}  // namespace lrfg
