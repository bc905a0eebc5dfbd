// fp64.cuh -- FP64 helpers. An SM issues two FP64 operations a cycle (16 cycles
// a warp instruction), so the small kernels that end in FP64 count them.
#pragma once

namespace game {

// x / m for a fixed divisor with r = 1 / m correctly rounded: one Newton
// correction of x r by its exact residual gives the correctly rounded quotient
// (Markstein, IBM J. Res. Dev. 34, 1990); the general division where the
// residual would not be exact. Three dependent operations instead of a
// division's dozen.
__device__ __forceinline__ double divide_by(double x, double m, double r) {
  const double ax = fabs(x);
  if (!(ax > 1e-250 && ax < 1e250)) return x / m;
  const double q = x * r;
  return fma(fma(-q, m, x), r, q);
}

}  // namespace game
