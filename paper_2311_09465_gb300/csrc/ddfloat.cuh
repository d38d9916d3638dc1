// Double-float ("float-float") arithmetic: a value is the unevaluated sum
// hi + lo of two FP32 numbers with |lo| <= ulp(hi)/2, about 48 significant
// bits.  Built from error-free transformations:
//   TwoSum (Knuth, TAOCP vol. 2, 4.2.2): s + e = a + b exactly;
//   FastTwoSum (Dekker 1971): the same when |a| >= |b|;
//   TwoProd with a fused multiply-add: p + e = a * b exactly.
// sqrt and the reciprocal take one Newton correction from the FP32 value.
// Sums carry an absolute error of about 2^-46 of the largest operand, which
// is what the element operator and the entries of tau's matrix need; the
// exponent range is FP32's.
#pragma once

namespace ts {

struct dd {
  float hi, lo;
};

__device__ __forceinline__ dd dd_from_double(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}

// The same without the FP64 pipe (each of its instructions costs as much issue
// time as dozens of integer ones): hi is x rounded to 24 bits (ties away from
// zero), lo the signed remainder of 28 bits rounded to FP32.  |x| below 2^-126
// gives 0; infinities and NaN pass through.
__device__ __forceinline__ dd dd_split(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)(b >> 52) & 0x7ff;                       // biased exponent
  if (e < 897) return {0.f, 0.f};
  if (e > 1149)                                               // FP32 overflow, infinity, NaN
    return {e == 0x7ff && (b << 12) ? __int_as_float(0x7fffffff) : __int_as_float((int)(sign | 0x7f800000u)), 0.f};
  // exponent e - 896, 23 bits of the mantissa; a carry moves into the exponent
  const unsigned h = (unsigned)((b + 0x10000000ull) >> 29) - 0xc0000000u;
  const int rem = (int)((unsigned)b << 3) >> 3;               // x - hi in units of 2^(e - 1075)
  const float unit = __int_as_float((int)(sign | ((unsigned)(e - 896) << 23)));   // 2^(e - 1023)
  return {__int_as_float((int)(h | sign)), ((float)rem * 2.220446049250313e-16f) * unit};
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  e = b - (s - a);
}

__device__ __forceinline__ dd dd_neg(dd a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ dd dd_add(dd a, dd b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e += a.lo + b.lo;
  dd r;
  fast_two_sum(s, e, r.hi, r.lo);
  return r;
}

// a * b + c
__device__ __forceinline__ dd dd_fma(dd a, dd b, dd c) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  float s, t;
  two_sum(p, c.hi, s, t);
  t += e + c.lo;
  dd r;
  fast_two_sum(s, t, r.hi, r.lo);
  return r;
}

__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  dd r;
  fast_two_sum(p, e, r.hi, r.lo);
  return r;
}

__device__ __forceinline__ dd dd_scale(dd a, float pow2) { return {a.hi * pow2, a.lo * pow2}; }

// sqrt(a) for a > 0: s0 = sqrt(hi), then s0 + (a - s0^2) / (2 s0)
__device__ __forceinline__ dd dd_sqrt(dd a) {
  const float s0 = sqrtf(a.hi);
  const float p = s0 * s0;
  const float e = fmaf(s0, s0, -p);
  const float rem = ((a.hi - p) - e) + a.lo;
  dd r;
  fast_two_sum(s0, rem / (2.f * s0), r.hi, r.lo);
  return r;
}

// 1 / a: y0 = 1/hi, then y0 + y0 (1 - a y0)
__device__ __forceinline__ dd dd_rcp(dd a) {
  const float y0 = 1.f / a.hi;
  const float p = a.hi * y0;
  const float e = fmaf(a.hi, y0, -p);
  const float rem = ((1.f - p) - e) - a.lo * y0;
  dd r;
  fast_two_sum(y0, y0 * rem, r.hi, r.lo);
  return r;
}

}  // namespace ts
