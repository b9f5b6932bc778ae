// Sums of float products as unevaluated sums of two or three floats (error-free products by a fused multiply-add and
// error-free additions by Knuth's TwoSum; Ogita, Rump and Oishi's Dot2 and DotK): the FP32 units do the
// work of FP64, whose instructions run at 1/64 of their rate here.
//
//   Pair     an error of n^2 2^-48 of the summands' absolute values, as if in twice the float precision
//   Triple   n^3 2^-72, then one rounding to double: for what must be no worse than a sum in double
//
// However many floats are added up, their exponents are a float's: square_exact() tells which squares, and rounding
// errors of squares, are representable.
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

// (h, l) += ph + pl, and += a x
__device__ __forceinline__ void pair_add(float& h, float& l, float ph, float pl) {
  float t, e;
  two_sum(h, ph, t, e);
  h = t;
  l = __fadd_rn(l, __fadd_rn(e, pl));
}
__device__ __forceinline__ void dot2(float& h, float& l, float a, float x) {
  const float p = __fmul_rn(a, x);
  pair_add(h, l, p, __fmaf_rn(a, x, -p));
}

struct Pair {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float ph, float pl) { pair_add(h, l, ph, pl); }
  __device__ __forceinline__ void fma(float a, float x) { dot2(h, l, a, x); }
  __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

struct Triple {
  float h = 0.f, l = 0.f, m = 0.f;
  __device__ __forceinline__ void low(float x) {   // += x, of the order of l
    float t, e;
    two_sum(l, x, t, e);
    l = t;
    m = __fadd_rn(m, e);
  }
  __device__ __forceinline__ void add(float x) {
    float t, e;
    two_sum(h, x, t, e);
    h = t;
    low(e);
  }
  __device__ __forceinline__ void add(float xh, float xl, float xm) {
    add(xh);
    low(xl);
    m = __fadd_rn(m, xm);
  }
  __device__ __forceinline__ void fma(float a, float x) {   // += a x
    const float p = __fmul_rn(a, x);
    add(p);
    low(__fmaf_rn(a, x, -p));
  }
  __device__ __forceinline__ void fma(float a, float xh, float xl, float xm) {   // += a (xh + xl + xm)
    fma(a, xh);
    const float q = __fmul_rn(a, xl);
    low(q);
    m = __fadd_rn(m, __fmaf_rn(a, xm, __fmaf_rn(a, xl, -q)));
  }
  __device__ __forceinline__ double value() const { return (double)h + ((double)l + (double)m); }
};

// A sum of squares of floats of any size, as accurate as one in double: those that leave the float range are added up in
// double.  N at a time, so that a check in between does not keep their loads apart.
struct Squares {
  Triple t;
  double rest = 0.0;
  template <int N>
  __device__ __forceinline__ void add(const float (&x)[N]) {
    bool all = true;
#pragma unroll
    for (int q = 0; q < N; ++q) all = all && square_exact(x[q]);
    if (all) {
#pragma unroll
      for (int q = 0; q < N; ++q) t.fma(x[q], x[q]);
    } else {
#pragma unroll
      for (int q = 0; q < N; ++q) {
        if (square_exact(x[q])) t.fma(x[q], x[q]);
        else rest += (double)x[q] * (double)x[q];
      }
    }
  }
  __device__ __forceinline__ double value() const { return t.value() + rest; }
};

}  // namespace dev
}  // namespace qrkit
