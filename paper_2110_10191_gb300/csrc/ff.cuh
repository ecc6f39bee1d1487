// ff.cuh -- float-float ("double-word") arithmetic on the FP32 pipe.
//
// A value is the unevaluated sum hi + lo of two floats with |lo| <= ulp(hi)/2,
// about 48 significant bits.  GB300 issues FP32 operations at 64 times the
// FP64 rate, so a float-float operation (5 to 20 FP32 instructions) costs a
// fraction of an FP64 one.  The building blocks are the error-free
// transformations of the literature, written here from their definitions:
//   two_sum       Knuth (TAOCP vol. 2, 4.2.2) / Moller (1965): s + e = a + b exactly
//   fast_two_sum  Dekker (1971): the same when |a| >= |b|
//   two_prod      with a fused multiply-add: p + e = a b exactly
// and the double-word algorithms analysed by Joldes, Muller and Popescu
// (ACM TOMS 2017): the "sloppy" sum (relative error bounded when both
// operands have the same sign; absolute error about 2^-47 (|a| + |b|)
// otherwise), the product with the cross terms folded into the FMA, and one
// Newton step in float-float for the reciprocal, the inverse square root
// (seeded by the hardware approximations on the high word) and the square
// root (seeded by the FP32 square root).
//
// Every primitive uses the _rn intrinsics, which the compiler never fuses
// into FMAs, so the error-free transformations stay exact.
#pragma once

#include <cuda_runtime.h>

#include "wide.cuh"

namespace grmhd {

struct ff {
  float hi, lo;
};

__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

__device__ __forceinline__ float fast_two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
  return s;
}

__device__ __forceinline__ ff ff_make(float hi, float lo) {
  ff r;
  r.hi = fast_two_sum(hi, lo, r.lo);
  return r;
}

// double -> float-float: the high word is x rounded to float, the low word
// the rounded remainder (48 of the 53 bits are kept).  The conversion
// instructions occupy the FP64 unit for 66 cycles each, which kernels with enough
// FP32 work beside them hide.
__device__ __forceinline__ ff ff_from(double x) {
  ff r;
  r.hi = __double2float_rn(x);
  r.lo = __double2float_rn(__dsub_rn(x, (double)r.hi));
  return r;
}

// Out of line, so that the compiler does not run the conversions beside the integer
// forms below in every thread and choose afterwards (a 128^3 state's split took 0.19
// ms so, 0.11 without).
static __device__ __noinline__ ff ff_from_call(double x) { return ff_from(x); }
static __device__ __noinline__ double f_to_double_call(float f) { return (double)f; }

// The same on the integer pipes where the high word is a normal float or zero: the
// bits taken apart, the remainder, 29 bits, converted as an integer and scaled in two
// steps of which only the last may round, to a subnormal (a tie of the high word may
// round the other way, the sum of the words stays the same).
__device__ __forceinline__ ff ff_from_bits(double x) {
  const u64 b = w_bits(x);
  const u32 sign = w_hi(b) & 0x80000000u;
  const int e = (int)((w_hi(b) >> 20) & 0x7ff);
  if (e < 873) return ff{__uint_as_float(sign), __uint_as_float(sign)};  // below float's last place
  if ((u32)(e - 897) >= 240u) return ff_from_call(x);
  const u64 m = (b & (~0ull >> 1)) + (1ull << 28);
  const int rest = (int)(w_lo(b) << 3) >> 3;  // x - hi in units of x's last place
  const float lo = __fmul_rn(__fmul_rn(__int2float_rn(rest), 0x1p-64f),
                             __int_as_float((e - 884) << 23));
  ff r;
  r.hi = __uint_as_float(((u32)(m >> 29) - (896u << 23)) | sign);
  r.lo = __uint_as_float(__float_as_uint(lo) ^ sign);
  return r;
}

// a float as a double, normal values and zeros by their bits
__device__ __forceinline__ double f_to_double(float f) {
  const u32 u = __float_as_uint(f), m = u & 0x7fffffffu;
  if (m != 0u && m - 0x800000u >= 0x7f000000u) return f_to_double_call(f);  // subnormal, infinite, NaN
  const u32 hi = (m ? (m >> 3) + (896u << 20) : 0u) | (u & 0x80000000u);
  return w_double((u64)hi << 32 | (u64)(u << 29));
}

// d 2^k for a result in the normal range
__device__ __forceinline__ double d_scale(double d, int k) {
  const u64 b = w_bits(d);
  const u32 f = (w_hi(b) >> 20) & 0x7ffu;
  return (f == 0u || f == 0x7ffu) ? d : w_double(b + ((u64)(s64)k << 52));
}

__device__ __forceinline__ ff ff_f(float x) {
  ff r;
  r.hi = x;
  r.lo = 0.0f;
  return r;
}

// float-float -> double, by the conversion instructions and by the bits
__device__ __forceinline__ double ff_to(ff a) { return __dadd_rn((double)a.hi, (double)a.lo); }
__device__ __forceinline__ double ff_to_bits(ff a) {
  return __dadd_rn(f_to_double(a.hi), f_to_double(a.lo));
}

__device__ __forceinline__ ff ff_neg(ff a) {
  ff r;
  r.hi = -a.hi;
  r.lo = -a.lo;
  return r;
}

// exact scaling by a power of two
__device__ __forceinline__ ff ff_ldexp(ff a, float p2) {
  ff r;
  r.hi = __fmul_rn(a.hi, p2);
  r.lo = __fmul_rn(a.lo, p2);
  return r;
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
  float e;
  const float s = two_sum(a.hi, b.hi, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return ff_make(s, e);
}

__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }

__device__ __forceinline__ ff ff_add_f(ff a, float b) {
  float e;
  const float s = two_sum(a.hi, b, e);
  e = __fadd_rn(e, a.lo);
  return ff_make(s, e);
}

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return ff_make(p, e);
}

__device__ __forceinline__ ff ff_mul_f(ff a, float b) {
  const float p = __fmul_rn(a.hi, b);
  float e = __fmaf_rn(a.hi, b, -p);
  e = __fmaf_rn(a.lo, b, e);
  return ff_make(p, e);
}

__device__ __forceinline__ ff ff_sqr(ff a) {
  const float p = __fmul_rn(a.hi, a.hi);
  float e = __fmaf_rn(a.hi, a.hi, -p);
  e = __fmaf_rn(__fmul_rn(2.0f, a.hi), a.lo, e);
  return ff_make(p, e);
}

// 1/a: FP32 seed r (the hardware approximation, within about an ulp of 1/hi; a is
// never near the float underflow in these bodies, which work in scaled units) and
// r + r (e + e^2) with e = 1 - a r, whose first product is exact in the FMA.  Worst
// relative error 2^-45.0 over seeds an ulp off, in 8 instructions: e as a
// float-float and without its square took 33 and left 2^-44.3.
__device__ __forceinline__ ff ff_rcp(ff a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a.hi));
  float e = __fmaf_rn(-a.hi, r, 1.0f);
  e = __fmaf_rn(-a.lo, r, e);
  return ff_make(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

__device__ __forceinline__ ff ff_div(ff a, ff b) { return ff_mul(a, ff_rcp(b)); }

// sqrt(a), a >= 0: s0 = sqrtf(hi), then s0 + (a - s0^2) / (2 s0)
__device__ __forceinline__ ff ff_sqrt(ff a) {
  if (!(a.hi > 0.0f)) return ff_f(0.0f);
  const float s0 = __fsqrt_rn(a.hi);
  float e;
  const float p = __fmul_rn(s0, s0);
  e = __fmaf_rn(s0, s0, -p);  // s0^2 = p + e exactly
  const ff d = ff_sub(a, ff_make(p, e));
  return ff_add_f(ff_mul_f(d, __fdiv_rn(0.5f, s0)), s0);
}

// 1/sqrt(a), a > 0: y from the hardware approximation of 1/sqrt(hi), then
// y + y (e/2 + 3 e^2/8) with e = 1 - a y^2 from the exact product hi y = p + q
// (worst relative error 2^-44.8 in 14 instructions; 2^-44.0 in 38 with e as a
// float-float to the first order)
__device__ __forceinline__ ff ff_rsqrt(ff a) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.hi));
  const float p = __fmul_rn(a.hi, y), q = __fmaf_rn(a.hi, y, -p);
  float e = __fmaf_rn(-p, y, 1.0f);
  e = __fmaf_rn(-q, y, e);
  e = __fmaf_rn(__fmul_rn(-a.lo, y), y, e);
  return ff_make(y, __fmul_rn(y, __fmaf_rn(__fmul_rn(0.375f, e), e, __fmul_rn(0.5f, e))));
}

__device__ __forceinline__ bool ff_gt(ff a, ff b) {
  return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo);
}
__device__ __forceinline__ ff ff_max(ff a, ff b) { return ff_gt(a, b) ? a : b; }
__device__ __forceinline__ ff ff_min(ff a, ff b) { return ff_gt(a, b) ? b : a; }
__device__ __forceinline__ ff ff_abs(ff a) { return (a.hi < 0.0f) ? ff_neg(a) : a; }

}  // namespace grmhd
