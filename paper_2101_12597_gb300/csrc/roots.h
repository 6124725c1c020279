// FP64 square roots and reciprocal square roots from a single-precision seed,
// for chains of dependent scalars (a correctly rounded root and a division take
// some 20 FP64 operations each).  Plain arithmetic, compiled for the device
// and, in the tests, for the host.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define ETDM_ROOTS_HD __host__ __device__ __forceinline__
#else
#define ETDM_ROOTS_HD inline
#endif

namespace etdm {

// y (3 - x y^2) / 2: a Newton-Raphson step of x^(-1/2), squares the relative error
ETDM_ROOTS_HD double root_step(double x, double y) { return y * fma(-0.5 * x, y * y, 1.5); }

// x^(-1/2) from a seed of relative error below 2^-21: one step, then a
// correction added last, so that its own rounding is the largest error (below
// 1 unit in the last place; a second step leaves 1.5, 1 / sqrt(x) 1.4)
ETDM_ROOTS_HD double root_rsqrt(double x, double seed) {
  const double y = root_step(x, seed), e = fma(-(x * y), y, 1.0);
  return fma(0.5 * e, y, y);
}

// x^(1/2), correctly rounded but for near-ties: y = x^(-1/2) to 2^-41, and the
// exact residual of s = x y
ETDM_ROOTS_HD double root_sqrt(double x, double seed) {
  const double y = root_step(x, seed), s = x * y;
  return fma(fma(-s, s, x), 0.5 * y, s);
}

}  // namespace etdm
