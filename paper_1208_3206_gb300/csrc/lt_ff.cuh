// lt_ff.cuh -- float-float arithmetic (an unevaluated sum of two FP32 numbers,
// about 46 bits) for quantities that need more than FP32 on a chip whose FP64
// pipe issues two lanes per clock and SM: one FP64 warp instruction occupies
// it for 16 clocks, a float-float product is 7 FP32 instructions (under 2
// clocks). Sums and products after Dekker (1971) and Knuth. Every operation
// is an explicitly rounded intrinsic, so that the compiler cannot contract or
// reorder the error terms.
#pragma once

namespace lt {

struct ff {
  float h, l;
};

__device__ __forceinline__ ff ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}

// |a| >= |b| (or a = 0)
__device__ __forceinline__ ff ff_fast_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ ff ff_two_diff(float a, float b) { return ff_two_sum(a, -b); }

__device__ __forceinline__ ff ff_two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}

// absolute error at most about 2^-46 (|a| + |b|)
__device__ __forceinline__ ff operator+(ff a, ff b) {
  const ff s = ff_two_sum(a.h, b.h);
  return ff_fast_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}

__device__ __forceinline__ ff operator-(ff a) { return {-a.h, -a.l}; }
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }

__device__ __forceinline__ ff operator+(ff a, float b) {
  const ff s = ff_two_sum(a.h, b);
  return ff_fast_sum(s.h, __fadd_rn(s.l, a.l));
}

// relative error about 2^-45
__device__ __forceinline__ ff operator*(ff a, ff b) {
  const ff p = ff_two_prod(a.h, b.h);
  return ff_fast_sum(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}

__device__ __forceinline__ ff operator*(ff a, float b) {
  const ff p = ff_two_prod(a.h, b);
  return ff_fast_sum(p.h, __fmaf_rn(a.l, b, p.l));
}

// a / b: FP32 quotient, then one correction from the float-float residual
// (relative error about 2^-44); b.h and the quotient well inside FP32 range
__device__ __forceinline__ ff operator/(ff a, ff b) {
  const float r = __frcp_rn(b.h);
  const float q = __fmul_rn(a.h, r);
  const ff res = a - b * q;
  const float q1 = __fmul_rn(__fadd_rn(res.h, res.l), r);
  return ff_fast_sum(q, q1);
}

__device__ __forceinline__ double ff_double(ff a) { return (double)a.h + (double)a.l; }

// (float)((double)acc * unit) for a 64-bit fixed-point sum, with the unit as a
// float-float pair: two exact 23-bit pieces of the sum times the pair, rounded
// once at the end. It can differ from the FP64 form only where that value lies
// within about 2^-44 of a rounding boundary; sums of 2^46 and more take FP64.
// In FP64 the conversion of a 512^3 grid was bound by the FP64 pipe (94% busy,
// 685 us for 1.6 GB).
struct FixedScale {
  ff u;         // unit
  double unit;  // the same in FP64
  bool small;   // the pair represents the unit (inside FP32's range with room)
};

__host__ __device__ inline FixedScale fixed_scale(double unit) {
  FixedScale s;
  s.unit = unit;
  s.u.h = (float)unit;
  s.u.l = (float)(unit - (double)s.u.h);
  s.small = unit > 1e-25 && unit < 1e20;
  return s;
}

__device__ __forceinline__ float fixed_to_float(unsigned long long acc, const FixedScale& s) {
  const unsigned hi = (unsigned)(acc >> 23);
  if (!s.small || (acc >> 46)) return (float)((double)acc * s.unit);
  // exact integers below 2^23 as floats: mantissa bits under the exponent of 2^23
  const float a = __fsub_rn(__uint_as_float(0x4b000000u | hi), 8388608.0f) * 8388608.0f;
  const float b = __fsub_rn(__uint_as_float(0x4b000000u | ((unsigned)acc & 0x7fffffu)), 8388608.0f);
  const ff n = ff_fast_sum(a, b);  // exact: a is a multiple of 2^23, b below it
  const ff p = ff_two_prod(n.h, s.u.h);
  return __fadd_rn(p.h, __fmaf_rn(n.h, s.u.l, __fmaf_rn(n.l, s.u.h, p.l)));
}

// (float)((double)acc * unit * factor), the same way.
__device__ __forceinline__ float fixed_to_float(unsigned long long acc, const FixedScale& s, float factor) {
  const unsigned hi = (unsigned)(acc >> 23);
  if (!s.small || (acc >> 46)) return (float)((double)acc * s.unit * (double)factor);
  const float a = __fsub_rn(__uint_as_float(0x4b000000u | hi), 8388608.0f) * 8388608.0f;
  const float b = __fsub_rn(__uint_as_float(0x4b000000u | ((unsigned)acc & 0x7fffffu)), 8388608.0f);
  const ff v = ff_fast_sum(a, b) * s.u;
  const ff p = ff_two_prod(v.h, factor);
  return __fadd_rn(p.h, __fmaf_rn(v.l, factor, p.l));
}

}  // namespace lt
