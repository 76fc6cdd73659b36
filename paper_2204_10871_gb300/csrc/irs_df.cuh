// irs_df.cuh -- double-float ("double-word") arithmetic on the FP32 pipes for
// the far-field convolution (FFTs and M2L).  A value is the unevaluated sum
// hi + lo of two floats with |lo| <= ulp(hi)/2: 48 significant bits.  GB300
// runs FP64 at 1/64 of its FP32 rate, and a double-float multiply-add costs
// ~30 FP32 operations, so the convolution moves to the FP32 pipes.
//
// The building blocks are the error-free transformations of Knuth (TwoSum),
// Dekker (Fast2Sum) and the FMA form of TwoProd; the sums and products follow
// the "sloppy" double-word addition and the double-word x double-word
// product of Joldes, Muller and Popescu (ACM TOMS 44, 2017), whose relative
// error is a few 2^-48 in the normwise sense an FFT needs.  Every operation
// goes through __fadd_rn / __fmul_rn / __fmaf_rn, so that the compiler cannot
// contract or reorder the exact-rounding steps.
#pragma once

#include <cuda_runtime.h>

namespace irs {

__device__ __forceinline__ void df_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// |a| >= |b| (or a == 0)
__device__ __forceinline__ void df_fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// x + y (sloppy double-word addition)
__device__ __forceinline__ float2 df_add(float2 x, float2 y) {
  float s, e, h, l;
  df_two_sum(x.x, y.x, s, e);
  e = __fadd_rn(e, __fadd_rn(x.y, y.y));
  df_fast_two_sum(s, e, h, l);
  return make_float2(h, l);
}

__device__ __forceinline__ float2 df_neg(float2 x) { return make_float2(-x.x, -x.y); }

__device__ __forceinline__ float2 df_sub(float2 x, float2 y) { return df_add(x, df_neg(y)); }

// x * y
__device__ __forceinline__ float2 df_mul(float2 x, float2 y) {
  const float p = __fmul_rn(x.x, y.x);
  float e = __fmaf_rn(x.x, y.x, -p);
  e = __fmaf_rn(x.x, y.y, e);
  e = __fmaf_rn(x.y, y.x, e);
  float h, l;
  df_fast_two_sum(p, e, h, l);
  return make_float2(h, l);
}

// Complex double-float, stored as float4 (re.hi, im.hi, re.lo, im.lo): the two
// parts' high words, and their low words, are register pairs, so that the sums
// go through the packed FP32x2 instructions, real and imaginary part at once
// (the same roundings in half the issue slots).  Products stay scalar, since their
// operands cross between the parts, up to the packed sum of the two products.
__device__ __forceinline__ float2 dfc_hi(float4 z) { return make_float2(z.x, z.y); }
__device__ __forceinline__ float2 dfc_lo(float4 z) { return make_float2(z.z, z.w); }
__device__ __forceinline__ float2 dfc_re(float4 z) { return make_float2(z.x, z.z); }
__device__ __forceinline__ float2 dfc_im(float4 z) { return make_float2(z.y, z.w); }
__device__ __forceinline__ float4 dfc_make(float2 re, float2 im) { return make_float4(re.x, im.x, re.y, im.y); }

// a - b: one rounding
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// high words s + e renormalised (Fast2Sum)
__device__ __forceinline__ float4 dfc_norm(float2 s, float2 e) {
  const float2 h = __fadd2_rn(s, e), l = sub2(e, sub2(h, s));
  return make_float4(h.x, h.y, l.x, l.y);
}

// x + y + lo for high words x, y (TwoSum)
__device__ __forceinline__ float4 dfc_sum(float2 x, float2 y, float2 lo) {
  const float2 s = __fadd2_rn(x, y), bb = sub2(s, x);
  const float2 e = __fadd2_rn(sub2(x, sub2(s, bb)), sub2(y, bb));
  return dfc_norm(s, __fadd2_rn(e, lo));
}

__device__ __forceinline__ float4 dfc_mul(float4 a, float4 b) {
  // a.re b.re - a.im b.im and a.re b.im + a.im b.re, each product as p + e
  float2 p1, e1, p2, e2;
  p1.x = __fmul_rn(a.x, b.x);
  p1.y = __fmul_rn(a.x, b.y);
  e1.x = __fmaf_rn(a.z, b.x, __fmaf_rn(a.x, b.z, __fmaf_rn(a.x, b.x, -p1.x)));
  e1.y = __fmaf_rn(a.z, b.y, __fmaf_rn(a.x, b.w, __fmaf_rn(a.x, b.y, -p1.y)));
  p2.x = __fmul_rn(-a.y, b.y);
  p2.y = __fmul_rn(a.y, b.x);
  e2.x = __fmaf_rn(-a.w, b.y, __fmaf_rn(-a.y, b.w, __fmaf_rn(-a.y, b.y, -p2.x)));
  e2.y = __fmaf_rn(a.w, b.x, __fmaf_rn(a.y, b.z, __fmaf_rn(a.y, b.x, -p2.y)));
  return dfc_sum(p1, p2, __fadd2_rn(e1, e2));
}

__device__ __forceinline__ float4 dfc_add(float4 a, float4 b) {
  return dfc_sum(dfc_hi(a), dfc_hi(b), __fadd2_rn(dfc_lo(a), dfc_lo(b)));
}

__device__ __forceinline__ float4 dfc_sub(float4 a, float4 b) {
  const float2 x = dfc_hi(a), y = dfc_hi(b);
  const float2 s = sub2(x, y), bb = sub2(s, x);
  const float2 e = sub2(sub2(x, sub2(s, bb)), __fadd2_rn(y, bb));
  return dfc_norm(s, __fadd2_rn(e, sub2(dfc_lo(a), dfc_lo(b))));
}

// x * s for a double-float real s
__device__ __forceinline__ float4 dfc_scale(float4 a, float2 s) {
  const float2 p = make_float2(__fmul_rn(a.x, s.x), __fmul_rn(a.y, s.x));
  float2 e;
  e.x = __fmaf_rn(a.z, s.x, __fmaf_rn(a.x, s.y, __fmaf_rn(a.x, s.x, -p.x)));
  e.y = __fmaf_rn(a.w, s.x, __fmaf_rn(a.y, s.y, __fmaf_rn(a.y, s.x, -p.y)));
  return dfc_norm(p, e);
}

// FP64 <-> double-float
__host__ __device__ __forceinline__ float2 df_from_double(double x) {
  const float h = (float)x;
  return make_float2(h, (float)(x - (double)h));
}
__host__ __device__ __forceinline__ double df_to_double(float2 x) { return (double)x.x + (double)x.y; }
__host__ __device__ __forceinline__ float4 dfc_from_double(double re, double im) {
  const float2 r = df_from_double(re), i = df_from_double(im);
  return make_float4(r.x, i.x, r.y, i.y);
}

}  // namespace irs
