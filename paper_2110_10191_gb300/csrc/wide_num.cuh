// wide_num.cuh -- floating numbers of 63-bit magnitude on the integer pipes.
//
// A Wide is (-1)^s m 2^x with m < 2^63.  A product costs three 32x32->64 bit
// multiply-adds and a few additions, a sum of products aligned to its largest
// exponent about ten instructions a term, where GB300 issues one FP64
// instruction per 76 cycles and sub-partition (wide.cuh).  Results are not
// rounded but truncated, at 2^-60 of the largest term or operand product, and
// are left unnormalised where the next operations have the bits to spare (each
// product of two such numbers costs two more): norm() where they have not.
// Truncations are of magnitudes, so that a change of sign of the operands
// changes only the sign of the result.
#pragma once

#include "wide.cuh"

namespace grmhd {

struct Wide {
  u64 m;
  int s;  // sign mask: 0 or -1
  int x;
};

// m in [2^62, 2^63); a subnormal keeps its value
WIDE_FN Wide wide(double d) {
  const u64 b = w_bits(d);
  const u32 h = w_hi(b);
  const int f = (int)((h >> 20) & 0x7ff);
  Wide r;
  r.m = (((u64)((h & 0xfffffu) | (f ? 0x100000u : 0u)) << 32) | w_lo(b)) << 10;
  r.s = (int)h >> 31;
  r.x = w_max(f, 1) - 1085;
  return r;
}
// the same for a positive normal d
WIDE_FN Wide wide_pos(double d) {
  const u64 b = w_bits(d);
  Wide r;
  r.m = ((b & 0xfffffffffffffull) | 1ull << 52) << 10;
  r.s = 0;
  r.x = (int)(w_hi(b) >> 20) - 1085;
  return r;
}
WIDE_FN bool w_finite(double d) { return (w_hi(w_bits(d)) & 0x7ff00000u) != 0x7ff00000u; }

// a b / 2^64 within 1 unit, for a, b < 2^63
WIDE_FN u64 w_mulhi63(u64 a, u64 b) {
  return w_mul(w_hi(a), w_hi(b)) + w_hi(w_mul(w_lo(a), w_hi(b)) + w_mul(w_hi(a), w_lo(b)));
}
WIDE_FN Wide operator*(const Wide &a, const Wide &b) {
  Wide r;
  r.m = w_mulhi63(a.m, b.m);  // < 2^62
  r.s = a.s ^ b.s;
  r.x = a.x + b.x + 64;
  return r;
}
WIDE_FN Wide operator-(const Wide &a) {
  Wide r = a;
  r.s = ~a.s;
  return r;
}
// a 2^k
WIDE_FN Wide w_scale(const Wide &a, int k) {
  Wide r = a;
  r.x += k;
  return r;
}
// m's top bit to bit 62, or 31 bits up where the upper word is zero (a sum that
// cancelled to 2^-30 of its terms has no use for more)
WIDE_FN Wide norm(const Wide &a) {
  const int k = w_clz32(w_hi(a.m)) - 1;
  Wide r;
  r.m = a.m << k;
  r.s = a.s;
  r.x = a.x - k;
  return r;
}

// Signed sums on the largest exponent, the magnitudes shifted right by H more
// bits so that the sum stays below 2^63: H = 0 for two products (each below
// 2^62), 1 for four products or two numbers, 2 for four numbers or one and four
// products.  A term is
// (m ^ s) - s; the s are gathered in one word.
WIDE_FN u64 w_term(const Wide &a, int x) { return w_shr(a.m, x - a.x) ^ (u64)(s64)a.s; }
WIDE_FN Wide w_sum_of(u64 terms, int s, int x) {
  const s64 S = (s64)terms - s;
  Wide r;
  r.s = (int)(S >> 32) >> 31;
  const u64 k = (u64)(s64)r.s;
  r.m = ((u64)S ^ k) - k;
  r.x = x;
  return r;
}
template <int H>
WIDE_FN Wide w_sum(const Wide &a, const Wide &b) {
  const int x = w_max(a.x, b.x) + H;
  return w_sum_of(w_term(a, x) + w_term(b, x), a.s + b.s, x);
}
template <int H>
WIDE_FN Wide w_sum(const Wide &a, const Wide &b, const Wide &c) {
  const int x = w_max(w_max(a.x, b.x), c.x) + H;
  return w_sum_of(w_term(a, x) + w_term(b, x) + w_term(c, x), a.s + b.s + c.s, x);
}
template <int H>
WIDE_FN Wide w_sum(const Wide &a, const Wide &b, const Wide &c, const Wide &d) {
  const int x = w_max(w_max(a.x, b.x), w_max(c.x, d.x)) + H;
  return w_sum_of(w_term(a, x) + w_term(b, x) + w_term(c, x) + w_term(d, x),
                  a.s + b.s + c.s + d.s, x);
}

template <int H>
WIDE_FN Wide w_sum(const Wide &a, const Wide &b, const Wide &c, const Wide &d, const Wide &e) {
  const int x = w_max(w_max(w_max(a.x, b.x), w_max(c.x, d.x)), e.x) + H;
  return w_sum_of(w_term(a, x) + w_term(b, x) + w_term(c, x) + w_term(d, x) + w_term(e, x),
                  a.s + b.s + c.s + d.s + e.s, x);
}

// the nearest double (the tail beyond 64 bits counted as zero); 0 below 2^-1022, infinite or
// not a number beyond the largest
WIDE_FN double w_to_double(const Wide &a) {
  const int k = w_clz64(a.m);
  const u64 m = a.m << (k & 63);
  const int f = a.x - k + (1023 + 63 - 1);  // exponent field, 1 below for m's own bit
  const u64 r = ((m >> 10) + 1) >> 1;
  u64 b = ((u64)(u32)w_min(f, 0x7fe) << 52) + r;
  if (f < 0 || a.m == 0) b = 0;
  return w_double(b | ((u64)(u32)(a.s & (int)0x80000000) << 32));
}

// 1 / sqrt(a) for a positive normalised a: the hardware's FP32 approximation y
// and the series (1 - h)^(-1/2) = 1 + h/2 + 3h^2/8 with h = 1 - a y^2 (below
// 2^-20; its third order, 5h^3/16, is left out) taken in 64 bits
WIDE_FN Wide w_rsqrt(const Wide &a) {
  // a = t 4^e, t in [1/4, 1) as tm / 2^64
  const int odd = a.x & 1;
  const u64 tm = a.m << odd;            // [2^62, 2^64)
  const int e = (a.x + 64 - odd) >> 1;  // a = tm 2^-64 2^(2e)
  const u32 th = w_hi(tm);
#ifdef __CUDA_ARCH__
  float y0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(__uint2float_rz(th)));
  const u32 y = __float2uint_rz(y0 * 0x1p38f);  // 2^22 / sqrt(t) in (2^22, 2^23]
#else
  const float y0 = 1.0f / __builtin_sqrtf((float)(th & 0xffffff00u));
  const u32 y = (u32)(y0 * 0x1p38f);
#endif
  const u64 y2 = w_mul(y, y) << 17;  // y^2 = 2^44 / t, below 2^47: <= 2^63
  // t y^2 2^17 / 2^64 = 2^61 (1 - h)
  const u64 ty = w_mul(w_hi(tm), w_hi(y2)) +
                 ((u64)w_hi(w_mul(w_hi(tm), w_lo(y2))) + w_hi(w_mul(w_lo(tm), w_hi(y2))));
  const s64 h = (s64)(1ull << 61) - (s64)ty;  // 2^61 h, below 2^41 in magnitude
  const int h1 = (int)(h >> 11);              // 2^50 h
#ifdef __CUDA_ARCH__
  const float hf = __fmul_rn(__int2float_rn(h1), 0x1p-50f);
  const int h2 = __float2int_rn(__fmul_rn(__fmul_rn(hf, hf), 0.75f * 0x1p58f));
#else
  const float hf = (float)h1 * 0x1p-50f;
  const int h2 = (int)__builtin_rintf(hf * hf * (0.75f * 0x1p58f));
#endif
  // y (1 + (h + 3h^2/4) / 2) on 2^(22 + 39)
  const s64 c = (s64)y * ((h >> 3) + h2);  // y (h + 3h^2/4) 2^58
  Wide r;
  r.m = (u64)(((s64)y << 39) + (c >> 20));  // (2^61, 2^62]
  r.s = 0;
  r.x = -e - 61;
  return r;
}

// 1 / a for a normalised a, at most 2^-57 low: 2^95 / h in 32 bits (w_rcp32) and
// one Newton step
WIDE_FN Wide w_rcp(const Wide &a) {
  const u64 h = a.m << 1;                // [2^63, 2^64)
  const u32 r = w_rcp32(w_hi(h)) - 2u;   // <= 2^95 / h, within 2^-28
  const u64 e = (1ull << 63) - (w_mul(r, w_hi(h)) + w_hi(w_mul(r, w_lo(h))));  // below 2^35
  Wide q;
  q.m = ((u64)r << 31) + (w_mul(r, (u32)(e >> 3)) >> 29);
  q.s = a.s;
  q.x = -125 - a.x;
  return q;
}

// a 2^k as a float (24 bits of the upper word); infinite beyond the largest, and no less
// than 2^-96 for a normalised a (what is smaller comes out larger)
WIDE_FN float w_to_float(const Wide &a, int k) {
  const int e = w_min(w_max(a.x + 32 + k, -126), 127);
#ifdef __CUDA_ARCH__
  const float f = __uint2float_rz(w_hi(a.m)) * __int_as_float((e + 127) << 23);
#else
  const float f = (float)(w_hi(a.m) & 0xffffff80u) * __builtin_ldexpf(1.0f, e);
#endif
  return a.s ? -f : f;
}
// a positive normal float
WIDE_FN Wide wide_posf(float f) {
#ifdef __CUDA_ARCH__
  const u32 b = __float_as_uint(f);
#else
  u32 b;
  memcpy(&b, &f, 4);
#endif
  Wide r;
  r.m = (u64)((b & 0x7fffffu) | 0x800000u) << 39;  // [2^62, 2^63)
  r.s = 0;
  r.x = (int)(b >> 23) - (127 + 62);
  return r;
}

}  // namespace grmhd
