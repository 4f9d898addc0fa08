// Float-float ("double-float") arithmetic: a value is the unevaluated sum
// hi + lo of two floats with |lo| <= ulp(hi)/2, about 48 significant bits.
//
// GB300 retires about two FP64 FMAs per clock per SM but 128 FP32 FMAs, so
// FP64-accurate FFT butterflies run faster as float-float on the FP32 pipes.
// The building blocks are the classical error-free transformations:
//   TwoSum (Knuth):        s = a + b exactly as s + e;
//   FastTwoSum (Dekker):   the same when |a| >= |b|;
//   TwoProduct with FMA:   a * b = p + e, e = fma(a, b, -p).
// Every operation uses the __f*_rn intrinsics so the compiler cannot
// contract or reassociate them (contraction would break the exactness of
// the error terms).  The addition is the "sloppy" variant: its error is
// bounded by about 2^-47 (|a| + |b|), which is the bound an FFT's error
// analysis uses anyway.
#pragma once

#include <cuda_runtime.h>

namespace aim {

struct ff {
  float hi, lo;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return ff{s, e};
}

__device__ __forceinline__ ff ff_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float e = __fsub_rn(b, __fsub_rn(s, a));
  return ff{s, e};
}

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return ff_fast_two_sum(p, e);
}

// acc + a * b with one closing renormalisation: the product's rounding
// error is recovered with FMA and carried in the low part, so the result is
// good to about 2^-47 (|acc| + |a b|).
__device__ __forceinline__ ff ff_mad(ff a, ff b, ff acc) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const ff s = ff_two_sum(acc.hi, p);
  const float t = __fadd_rn(__fadd_rn(s.lo, acc.lo), e);
  return ff_fast_two_sum(s.hi, t);
}

__device__ __forceinline__ ff ff_from_double(double v) {
  const float hi = __double2float_rn(v);
  const float lo = __double2float_rn(v - (double)hi);
  return ff{hi, lo};
}

// ------------------------------------------------------------------ two parts at a time
// Two FP32 operations in one instruction (f32x2, each half rounded to
// nearest).  The FP32 pipes' lane rate is the same for both forms (39 T lane
// operations/s measured), so what the packed form buys is issue slots and
// instruction-cache room: half the instructions of a complex addition or of a
// product with a real number.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 both(float c) { return make_float2(c, c); }
// a - b as one instruction (the product with -1 is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, both(-1.f), a); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }

// Complex float-float with its real and imaginary parts side by side:
// hi = (re.hi, im.hi), lo = (re.lo, im.lo), so each step of a two-sum or a
// two-product is one packed instruction for both parts.  Stored the same way
// (float4 = re.hi, im.hi, re.lo, im.lo).
struct cff2 {
  float2 hi, lo;
};
__device__ __forceinline__ cff2 cff2_ld(const float4& s) { return cff2{make_float2(s.x, s.y), make_float2(s.z, s.w)}; }
__device__ __forceinline__ float4 cff2_st(const cff2& t) { return make_float4(t.hi.x, t.hi.y, t.lo.x, t.lo.y); }
__device__ __forceinline__ cff2 cff2_zero() { return cff2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
__device__ __forceinline__ cff2 cff2_neg(cff2 a) { return cff2{neg2(a.hi), neg2(a.lo)}; }
__device__ __forceinline__ cff2 two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  const float2 bb = sub2(s, a);
  return cff2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ cff2 fast_two_sum2(float2 a, float2 b) {
  const float2 s = add2(a, b);
  return cff2{s, sub2(b, sub2(s, a))};
}
// Sums, sums of two products and ff_mad of each part.  The lazy sum leaves out
// the closing renormalisation: hi is the rounded sum of the high parts and lo
// collects that rounding error plus both low parts, so hi + lo still carries the
// sum to about 2^-47 (|a| + |b|) but |lo| may exceed ulp(hi)/2 by a few units.
// Later TwoSum/TwoProduct steps accept such pairs; used inside FFT butterflies,
// where every value feeds further arithmetic.
__device__ __forceinline__ cff2 cff2_add(cff2 a, cff2 b) {
  const cff2 s = two_sum2(a.hi, b.hi);
  return fast_two_sum2(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ cff2 cff2_add_lazy(cff2 a, cff2 b) {
  const cff2 s = two_sum2(a.hi, b.hi);
  return cff2{s.hi, add2(s.lo, add2(a.lo, b.lo))};
}
__device__ __forceinline__ cff2 cff2_dot2(cff2 a, cff2 b, cff2 c, cff2 d) {  // a b + c d, part by part
  const float2 p1 = mul2(a.hi, b.hi), p2 = mul2(c.hi, d.hi);
  const cff2 s = two_sum2(p1, p2);
  float2 e = fma2(a.hi, b.hi, neg2(p1));
  e = add2(e, fma2(c.hi, d.hi, neg2(p2)));
  e = fma2(a.hi, b.lo, e);
  e = fma2(a.lo, b.hi, e);
  e = fma2(c.hi, d.lo, e);
  e = fma2(c.lo, d.hi, e);
  e = add2(e, s.lo);
  return fast_two_sum2(s.hi, e);
}
__device__ __forceinline__ cff2 cff2_mad(cff2 a, cff2 b, cff2 acc) {  // acc + a b, part by part
  const float2 p = mul2(a.hi, b.hi);
  float2 e = fma2(a.hi, b.hi, neg2(p));
  e = fma2(a.hi, b.lo, e);
  e = fma2(a.lo, b.hi, e);
  const cff2 s = two_sum2(acc.hi, p);
  return fast_two_sum2(s.hi, add2(add2(s.lo, acc.lo), e));
}
// the same real number in both parts; i times a complex number
__device__ __forceinline__ cff2 cff2_both(ff r) { return cff2{both(r.hi), both(r.lo)}; }
__device__ __forceinline__ cff2 cff2_re(cff2 a) { return cff2{both(a.hi.x), both(a.lo.x)}; }
__device__ __forceinline__ cff2 cff2_im(cff2 a) { return cff2{both(a.hi.y), both(a.lo.y)}; }
__device__ __forceinline__ cff2 cff2_times_i(cff2 a) {
  return cff2{make_float2(-a.hi.y, a.hi.x), make_float2(-a.lo.y, a.lo.x)};
}
__device__ __forceinline__ cff2 cff2_shfl_xor(cff2 a, int o, int width) {
  return cff2{make_float2(__shfl_xor_sync(0xffffffffu, a.hi.x, o, width), __shfl_xor_sync(0xffffffffu, a.hi.y, o, width)),
              make_float2(__shfl_xor_sync(0xffffffffu, a.lo.x, o, width), __shfl_xor_sync(0xffffffffu, a.lo.y, o, width))};
}

}  // namespace aim
