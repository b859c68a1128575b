// FP64 reciprocal for the reflectors of the projected problem.
#pragma once

namespace lslu {

// 1 / d for 2^-1000 <= d <= 2^1000 from the hardware's approximation r, by one
// step of Chebyshev's method r - f/f' - f'' f^2 / (2 f'^3) for f(r) = 1/r - d:
// with e = 1 - d r it is r + r e + r e^2, the first terms of r / (1 - e) = 1/d.
// An e of 2^-20 leaves e^3 = 2^-60 and the rounding of the last sum: at most
// 0.51 units of the last place in all (0.506 measured), where a division has
// 0.5 and takes a step of the bidiagonalisation, which has two, 330 cycles more.
__device__ __forceinline__ double reciprocal(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  const double e = fma(-d, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace lslu
