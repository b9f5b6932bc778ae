// Sums of float products as unevaluated sums of two floats (error-free products by a fused multiply-add and
// error-free additions by Knuth's TwoSum; Ogita, Rump and Oishi's Dot2): the FP32 units do the
// work of FP64, whose instructions run at 1/64 of their rate here.  However many floats are added up, their exponents
// are a float's: square_exact() tells which squares, and rounding errors of squares, are representable.
#pragma once

#include <cuda_runtime.h>

#include "device_util.cuh"

namespace qrkit {
namespace dev {

// x = 0 or 2^-50 <= |x| <= 2^50: x^2 and its rounding error are exact in float, and 2^27 of them do not overflow.
// False for infinities and NaN.
__device__ __forceinline__ bool square_exact(float x) {
  const unsigned a = __float_as_uint(x) & 0x7fffffffu;
  return a - 1u >= ((127u - 50u) << 23) - 1u && a <= (127u + 50u) << 23;
}

struct Pair {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float ph, float pl) {   // += ph + pl
    float t, e;
    two_sum(h, ph, t, e);
    h = t;
    l = __fadd_rn(l, __fadd_rn(e, pl));
  }
  __device__ __forceinline__ void add(const Pair& o) { add(o.h, o.l); }
  __device__ __forceinline__ void fma(float a, float x) {   // += a x
    const float p = __fmul_rn(a, x);
    add(p, __fmaf_rn(a, x, -p));
  }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

}  // namespace dev
}  // namespace qrkit
