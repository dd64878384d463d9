// Reciprocal of a double for chains of pivots (host and device code).
#pragma once

#include <cmath>

#ifndef CLR_HD
#ifdef __CUDACC__
#define CLR_HD __host__ __device__
#else
#define CLR_HD
#endif
#endif

namespace clr {

// 1 / d to within one unit in the last place.  On the device: the hardware's ~2^-20 approximation and
// one third-order step y (1 + e + e^2), e = 1 - d y (Householder's method): three dependent FMAs, 213
// clocks in the place of a division's 569.  Outside 1e-290 < |d| < 1e290 (the approximation flushes
// subnormals) and on the host the division itself.
CLR_HD inline double near_rcp(double d) {
#ifdef __CUDA_ARCH__
  const double m = fabs(d);
  if (m > 1e-290 && m < 1e290) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
  }
#endif
  return 1.0 / d;
}

}  // namespace clr
