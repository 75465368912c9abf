// Sums of products of FP32 numbers to FP64 accuracy on the FP32 pipe (GB300's FP64
// pipe has 1/64 of its rate).  A sum is held in three words: the products enter as
// p + e exactly (TwoProduct by FMA; Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26
// (2005)), p joins the first word and what that loses (Knuth's TwoSum) the second
// together with e; what the second loses joins the third.  Only the third is rounded:
// n products err by at most 4 n^2 (n + 1) 2^-72 of their absolute sum, 2^-61 for
// eight, and converting the words to FP64 adds two roundings of 2^-53, where FP64
// multiply-adds take one per product.  Two sums run side by side (f32x2).
//
// Measured: a batch of 8^3 x 16 and three more lattices 172.6 -> 173.1 ms with this in
// the residual norms and in <p, q>.
//
// The products must neither overflow nor, where they count, lose bits below 2^-126:
// the operands are first scaled by a power of two (unit_exponent), exactly.
#pragma once

#include <cuda_runtime.h>

namespace bri {

struct Sum3 {
  float2 a, b, c;
};
__device__ __forceinline__ Sum3 sum3_zero() { return Sum3{make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
// s + e = s0 + v exactly; returns e
__device__ __forceinline__ float2 sum3_join(float2& s, float2 v) {
  const float2 t = __fadd2_rn(s, v);
  const float2 w = __fadd2_rn(t, make_float2(-s.x, -s.y));
  const float2 r = __fadd2_rn(t, make_float2(-w.x, -w.y));
  const float2 e = __fadd2_rn(__fadd2_rn(s, make_float2(-r.x, -r.y)), __fadd2_rn(v, make_float2(-w.x, -w.y)));
  s = t;
  return e;
}
// sum += x y
__device__ __forceinline__ void sum3_add(Sum3& s, float2 x, float2 y) {
  const float2 p = __fmul2_rn(x, y);
  const float2 e = __ffma2_rn(x, y, make_float2(-p.x, -p.y));
  const float2 u = sum3_join(s.b, sum3_join(s.a, p));
  const float2 v = sum3_join(s.b, e);
  s.c = __fadd2_rn(s.c, __fadd2_rn(u, v));
}
__device__ __forceinline__ double sum3_total(const Sum3& s) {
  return ((double)s.a.x + ((double)s.b.x + (double)s.c.x)) + ((double)s.a.y + ((double)s.b.y + (double)s.c.y));
}

// k such that 2^k v has a norm near 1 for a vector v of norm^2 n2; 2^k as a float and
// 2^-2k, the factor of its squares, as a double.
__device__ __forceinline__ int unit_exponent(double n2) {
  const int e = (int)((__double_as_longlong(n2) >> 52) & 2047) - 1023;  // (FP64 subnormals: the clamp)
  return max(-126, min(126, -(e >> 1)));
}
__device__ __forceinline__ float exp2_float(int k) { return __int_as_float((k + 127) << 23); }
__device__ __forceinline__ double exp2_square(int k) { return __longlong_as_double((long long)(1023 - 2 * k) << 52); }

}  // namespace bri
