// Two floats at a time (the f32x2 instructions): half the issue slots of the scalar forms at the same rate.
#pragma once

#include <cuda_runtime.h>

namespace qrkit {
namespace dev {

using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float x, float y) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ void unpack2(f2 d, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(d));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float sum2(f2 d) {
  float x, y;
  unpack2(d, x, y);
  return x + y;
}

// s + e = a + b exactly, in both halves (Knuth's TwoSum).
__device__ __forceinline__ void two_sum2(f2 a, f2 b, f2& s, f2& e) {
  s = add2(a, b);
  const f2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// The rounded product for an addition that needs it as such: a mul.rn.f32x2 (or an fma with a zero addend) and the
// add.rn.f32x2 that follows come out as one fma, which a Dot2 sum does not survive; two scalar mul.rn do not.
__device__ __forceinline__ f2 product2(f2 a, f2 b) {
  float a0, a1, b0, b1;
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  return pack2(__fmul_rn(a0, b0), __fmul_rn(a1, b1));
}

// (h, l) += a x by Dot2 (the product's and the sum's rounding errors are added to l), nx = -x.
__device__ __forceinline__ void dot2_add2(f2& h, f2& l, f2 a, f2 x, f2 nx) {
  const f2 p = product2(a, x), pe = fma2(a, x, mul2(a, nx));
  f2 s, e;
  two_sum2(h, p, s, e);
  h = s;
  l = add2(l, add2(e, pe));
}
// (h, l) += a (x + xl)
__device__ __forceinline__ void dot2_add2(f2& h, f2& l, f2 a, f2 x, f2 nx, f2 xl) {
  const f2 p = product2(a, x), pe = fma2(a, xl, fma2(a, x, mul2(a, nx)));
  f2 s, e;
  two_sum2(h, p, s, e);
  h = s;
  l = add2(l, add2(e, pe));
}

}  // namespace dev
}  // namespace qrkit
