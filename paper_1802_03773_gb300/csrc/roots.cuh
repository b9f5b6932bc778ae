// Roots and reciprocals of the Householder reflectors: the norm of a column and the inverses that tau and the
// scale need, by Newton's iteration with fused residuals (Newton-Raphson; Muller et al., Handbook of Floating-Point
// Arithmetic, "software implementation of division and square root").
//
// A reflector is orthogonal only as far as its tau is 2 / v^T v: a seed's error of one to two units in the last place has a
// sign of its own, and a row of R that meets dozens of reflectors drifts by as many of them.  One step
// from the hardware's seed brings the error below rounding, at a handful of multiply-adds.
#pragma once

#include <cuda_runtime.h>

namespace qrkit {
namespace dev {

// The root r of x >= 0 from a seed y of 1 / sqrt(x), r = x y + (x - (x y)^2) y / 2: within one unit in the last place (an
// infinite x gives itself).  The residual of a subnormal x is not representable: its root is CUDA's.
template <typename T>
__device__ __forceinline__ T newton_root(T x, T y) {
  constexpr T tiny = sizeof(T) == 4 ? T(1.17549435e-38) : T(2.2250738585072014e-308);   // the smallest normal number
  if (x < tiny) return sqrt(x);
  const T r = x * y;
  return y == T(0) ? x : fma(fma(-r, r, x), T(0.5) * y, r);
}
// 1 / x from a seed y: y + (1 - x y) y, within one unit in the last place (and 1 / infinity = 0).
template <typename T>
__device__ __forceinline__ T newton_inverse(T x, T y) {
  return y == T(0) ? y : fma(fma(-x, y, T(1)), y, y);
}

}  // namespace dev
}  // namespace qrkit
