// Roots and reciprocals of the Householder reflectors: the norm of a column and the inverses that tau and the
// scale need, by Newton's iteration with fused residuals (Newton-Raphson; Muller et al., Handbook of Floating-Point
// Arithmetic, "software implementation of division and square root").
//
// A reflector is orthogonal only as far as its tau is 2 / v^T v: a seed's error of one to two units in the last place has a
// sign of its own, and a row of R that meets dozens of reflectors drifts by as many of them.  One step
// from the hardware's seed brings the error below rounding, at a handful of multiply-adds.
#pragma once

#include <cuda_runtime.h>

#include "sums.cuh"

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
// The root of a sum h + l + m of floats (h the sum rounded, normal) in double: the float root of h, its remainder, which
// is a float, and two quotients of what is left.
__device__ __forceinline__ double root_of_sum(float h, float l, float m) {
  const float r = sqrtf(h);
  const float e = fmaf(-r, r, h);              // exact
  const float a = e + l, b = a - e;            // a + al = e + l (TwoSum)
  const float al = (e - (a - b)) + (l - b) + m;
  const float c = a / (2.f * r);
  const float d = (fmaf(-2.f * r, c, a) + fmaf(-c, c, al)) / (2.f * r);
  return (double)r + ((double)c + (double)d);
}
// sqrt(x^2 + y^2) of floats in double, to its last bits, with a quarter of the FP64 instructions (their squares as a sum
// of floats); in double where a square leaves the float range.
__device__ __forceinline__ double norm_of_two(float x, float y) {
  if (square_exact(x) && square_exact(y) && (x != 0.f || y != 0.f)) {
    Triple s;
    s.fma(x, x);
    s.fma(y, y);
    return root_of_sum(s.h, s.l, s.m);
  }
  return sqrt((double)x * (double)x + (double)y * (double)y);
}
// 1 / x from a seed y: y + (1 - x y) y, within one unit in the last place (and 1 / infinity = 0).
template <typename T>
__device__ __forceinline__ T newton_inverse(T x, T y) {
  return y == T(0) ? y : fma(fma(-x, y, T(1)), y, y);
}

}  // namespace dev
}  // namespace qrkit
