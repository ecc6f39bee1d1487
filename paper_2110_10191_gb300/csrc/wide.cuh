// wide.cuh -- WENO5 reconstruction in 64-bit integer arithmetic.
//
// GB300 issues one FP64 instruction per SM sub-partition every 76 cycles, a
// 32x32->64 bit multiply-add every 5, a 64-bit shift every 4 and a 64-bit
// addition every 2 (measured with one op per loop), so that an aligned sum
// (about 16 cycles) or a 60-bit product (about 18) costs a quarter of an FP64
// instruction.  The nonlinear weights and the weighted sum of a WENO5 pair are
// formed here that way: numbers are m 2^x with a 64-bit m, carried at 55 or
// more significant bits where FP64 rounds every operation to 53.
//
// The FP64 form of the pair (44.6 FP64 instructions per zone and primitive) was
// bound by that unit at any occupancy: 1.48 ms per direction on a 128^3 grid.
// Here three FP64 instructions remain (a first difference, the two final
// additions), the integer pipes bind, and the 128^3 WENO5 cycle went from 19.5
// to 13.8 ms.  Errors against exact arithmetic are no larger than FP64's (over
// random, smooth and jumping stencils: worst 4.3e-16 of the largest magnitude
// over both faces, 8.4e-16 in FP64).
//
// Every truncation is of a magnitude and every signed sum is exact, so that a
// mirrored stencil gives the same two face values swapped, bit for bit, and a
// stencil of the opposite sign the opposite values.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define WIDE_FN __host__ __device__ __forceinline__
#else
#define WIDE_FN inline
#endif

namespace grmhd {

typedef unsigned long long u64;
typedef long long s64;
typedef uint32_t u32;

WIDE_FN u32 w_hi(u64 a) { return (u32)(a >> 32); }
WIDE_FN u32 w_lo(u64 a) { return (u32)a; }
WIDE_FN u64 w_mul(u32 a, u32 b) { return (u64)a * b; }

WIDE_FN u64 w_bits(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
WIDE_FN double w_double(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((s64)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
WIDE_FN double w_fma(double a, double b, double c) {
#ifdef __CUDA_ARCH__
  return fma(a, b, c);
#else
  return __builtin_fma(a, b, c);
#endif
}
WIDE_FN int w_clz32(u32 a) {
#ifdef __CUDA_ARCH__
  return __clz((int)a);
#else
  return a ? __builtin_clz(a) : 32;
#endif
}
WIDE_FN int w_clz64(u64 a) {
#ifdef __CUDA_ARCH__
  return __clzll((s64)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}
WIDE_FN int w_min(int a, int b) { return a < b ? a : b; }
WIDE_FN int w_max(int a, int b) { return a > b ? a : b; }
// a >> n for 0 <= n, 0 when n > 63 (the PTX shift saturates its count)
WIDE_FN u64 w_shr(u64 a, int n) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
#else
  return n > 63 ? 0 : a >> n;
#endif
}
// sign mask (0 or -1), magnitude of a signed value, value of a magnitude
WIDE_FN s64 w_sign(s64 a) { return a >> 63; }
WIDE_FN u64 w_abs(s64 a, s64 s) { return (u64)((a ^ s) - s); }
WIDE_FN s64 w_signed(u64 m, s64 s) { return ((s64)m ^ s) - s; }

// a b / 2^64 and a^2 / 2^64, at most 2 and 1 units low (the low words'
// products are left out)
WIDE_FN u64 w_mulhi(u64 a, u64 b) {
  const u64 t = w_mul(w_hi(a), w_lo(b)), u = w_mul(w_lo(a), w_hi(b));
  return w_mul(w_hi(a), w_hi(b)) + ((u64)w_hi(t) + w_hi(u));
}
// the same within 1 unit for a < 2^61 and b < 2^63 (the middle sum fits)
WIDE_FN u64 w_mulhi61(u64 a, u64 b) {
  return w_mul(w_hi(a), w_hi(b)) + w_hi(w_mul(w_lo(a), w_hi(b)) + w_mul(w_hi(a), w_lo(b)));
}
WIDE_FN u64 w_sqrhi(u64 a) {
  return w_mul(w_hi(a), w_hi(a)) + (w_mul(w_hi(a), w_lo(a)) >> 31);
}

// 2^63 / a for a >= 2^31, at most 2 units low and never high: the hardware's
// FP32 approximation g of 2^55 / a and one Newton step, whose residual
// 2^55 - a g (below 2^34) is taken in 64 bits and its product in FP32
WIDE_FN u32 w_rcp32(u32 a) {
#ifdef __CUDA_ARCH__
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint2float_rz(a)));
  const u32 g = __float2uint_rz(f * 0x1p55f);
  const s64 e = (s64)(1ull << 55) - (s64)w_mul(a, g);
  const int c = __float2int_rd(__fmul_rn(__int2float_rz((int)(e >> 8)), __fmul_rn(f, 0x1p16f)));
#else
  const float f = 1.0f / (float)(a & 0xffffff00u);
  const u32 g = (u32)(f * 0x1p55f);
  const s64 e = (s64)(1ull << 55) - (s64)w_mul(a, g);
  const int c = (int)__builtin_floorf((float)(int)(e >> 8) * (f * 0x1p16f));
#endif
  return (g << 8) + (u32)c - 1u;
}

// One first difference: m 2^x with m of 60 bits; a subnormal keeps its value
// and zero has m = 0; an infinity or NaN has x = WIDE_X_BAD
struct WideDiff {
  u64 m;
  s64 s;  // sign mask
  int x;
};
constexpr int WIDE_X_BAD = 0x7ff - 1082;

WIDE_FN WideDiff wide_diff(double d) {
  const u64 b = w_bits(d);
  const u32 h = w_hi(b);
  const int f = (int)((h >> 20) & 0x7ff);
  const u32 mh = (h & 0xfffffu) | (f ? 0x100000u : 0u);
  WideDiff r;
  r.m = (((u64)mh << 32) | w_lo(b)) << 7;
  r.s = (s64)(int)h >> 31;
  r.x = w_max(f, 1) - 1082;
  return r;
}

// Two neighbouring first differences (a below, b above) on a common exponent,
// with the smoothness indicators of the substencil they span as seen from its
// three roles.  A substencil's 12 beta = 13 D^2 + 3 s^2 with D = b - a and s =
// 3b - a where it is the zone's lowest, a + b the middle and 3a - b the highest.
// Along a column, one new pair serves three zones.
struct WidePair {
  s64 a, b;  // |a|, |b| < 2^60
  int x;
};
struct WideNum {
  u64 m;
  int x;
};

WIDE_FN WidePair wide_pair(const WideDiff &a, const WideDiff &b) {
  WidePair p;
  p.x = w_max(a.x, b.x);
  p.a = w_signed(w_shr(a.m, p.x - a.x), a.s);
  p.b = w_signed(w_shr(b.m, p.x - b.x), b.s);
  return p;
}

// 12 eps = 1.2e-25 as m 2^WIDE_EPS_X
constexpr u64 WIDE_EPS_M = 1338044711911837388ull;
constexpr int WIDE_EPS_X = -143;

// (12 eps + 12 beta)^2 of a substencil, from its 13 D^2 and s on exponent x
// of the pair: m in [2^62, 2^64)
WIDE_FN WideNum wide_weight(u64 D13, s64 s, int x) {
  const u64 sq = w_sqrhi(w_abs(s, w_sign(s)));
  const u64 F = D13 + sq + (sq << 1);  // at most 25 * 2^58
  const int xf = 2 * x + 64, xe = w_max(xf, WIDE_EPS_X);
  const u64 e = w_shr(F, xe - xf) + w_shr(WIDE_EPS_M, xe - WIDE_EPS_X);  // 2^54 < e < 2^63
  const int n = w_clz32(w_hi(e));
  WideNum q;
  q.m = w_sqrhi(e << n);
  q.x = 2 * (xe - n);
  return q;
}

WIDE_FN u64 wide_D13(const WidePair &p) {
  const s64 D = p.b - p.a;
  const u64 d2 = w_sqrhi(w_abs(D, w_sign(D)));
  return 13 * d2;
}
WIDE_FN WideNum wide_q_low(const WidePair &p, u64 D13) { return wide_weight(D13, 3 * p.b - p.a, p.x); }
WIDE_FN WideNum wide_q_mid(const WidePair &p, u64 D13) { return wide_weight(D13, p.a + p.b, p.x); }
WIDE_FN WideNum wide_q_high(const WidePair &p, u64 D13) { return wide_weight(D13, 3 * p.a - p.b, p.x); }

// N / H 2^x as a double (rounded to nearest but for 2^-4 ulp; 0 below 2^-1022), for H >= 2^54
// and bad: NaN.  Both are normalised, h in [2^63, 2^64) and n in [2^62, 2^63),
// and n / h = (q0 + f) / 2^31 comes in two digits from r <= 2^95 / h: q0 = n r
// (at most 4.5 low) and f from the remainder n 2^31 - q0 h.
WIDE_FN double wide_quot(s64 N, u64 H, int x, bool bad) {
  const s64 sn = w_sign(N);
  const u64 a = w_abs(N, sn);
  const int kh = w_clz32(w_hi(H)), kn = w_clz64(a | 1u);
  const u64 h = H << kh, n = (a << kn) >> 1;
  const u32 r = w_rcp32(w_hi(h)) - 2u;  // 2: h's low word
  const u32 q0 = w_hi(w_mul(w_hi(n), r));
  const u64 rem = (n >> 1) - (w_mul(q0, w_hi(h)) + w_hi(w_mul(q0, w_lo(h))));  // < 4.5 2^32
  const u32 q1 = w_hi(w_mul((u32)(rem >> 3), r));  // f 2^28
  const u64 q = ((u64)q0 << 32) + ((u64)q1 << 4);  // n / h 2^63, in [2^61 - 2^34, 2^63)
  const int k = w_clz32(w_hi(q) | 1u);             // 1, 2 or (next to 2^61) 3
  const u64 m = ((q >> (10 - k)) + 1) >> 1;        // 53 bits, or 2^53
  const int f = x + kh - kn - k + 1023;          // exponent field, 1 below for m's own bit
  u64 b = ((u64)(u32)w_min(f, 0x7fe) << 52) + m;
  if (f < 0 || a == 0) b = 0;
  if (bad) b = 0x7ffull << 52 | 1ull << 51;
  return w_double(b | ((u64)sn & (1ull << 63)));
}

// Both WENO5 face values of a zone c from the pairs of first differences of
// its three substencils, lowest first, and their squared indicators: with W_0
// : W_1 : W_2 = q1 q2 : q0 q2 : q0 q1,
//   6 (hi - c) = (W_0 A + 6 W_1 B + 3 W_2 C) / (W_0 + 6 W_1 + 3 W_2),
//   6 (lo - c) = (W_2 A' - 6 W_1 B' - 3 W_0 C') / (3 W_0 + 6 W_1 + W_2),
// where the candidates' offsets are A = 5b - 2a, C' = 4b - a (lowest pair),
// B = a + 2b, B' = 2a + b (middle), C = 4a - b, A' = 2b - 5a (highest).
WIDE_FN void weno5_wide(double c, const WidePair &p0, const WidePair &p1, const WidePair &p2,
                        const WideNum &q0, const WideNum &q1, const WideNum &q2, double &lo,
                        double &hi) {
  const u64 w0 = w_mulhi(q1.m, q2.m), w1 = w_mulhi(q0.m, q2.m), w2 = w_mulhi(q0.m, q1.m);
  const int y0 = q1.x + q2.x, y1 = q0.x + q2.x, y2 = q0.x + q1.x;  // w >= 2^60
  // half the denominators, on exponent y + 4
  const int y = w_max(y0, w_max(y1, y2));
  const u64 g0 = w_shr(w0, y - y0 + 3), g1 = w_shr(w1, y - y1 + 3), g2 = w_shr(w2, y - y2 + 3);
  const u64 t1 = g1 + (g1 << 1);
  const u64 H = t1 + ((g0 + g2 + (g2 << 1)) >> 1), L = t1 + ((g2 + g0 + (g0 << 1)) >> 1);
  // the numerators, on exponent z + 3
  const int z0 = y0 + p0.x, z1 = y1 + p1.x, z2 = y2 + p2.x;
  const int z = w_max(z0, w_max(z1, z2));
  const u64 u0 = w_shr(w0, z - z0 + 3), u1 = w_shr(w1, z - z1 + 3), u2 = w_shr(w2, z - z2 + 3);
#define WIDE_TERM(w, v) w_signed(w_mulhi61(w, w_abs(v, w_sign(v))), w_sign(v))
  const s64 A = p0.b + (p0.b << 2) - (p0.a << 1), Cl = (p0.b << 2) - p0.a;
  const s64 B = p1.a + (p1.b << 1), Bl = (p1.a << 1) + p1.b;
  const s64 C = (p2.a << 2) - p2.b, Al = (p2.b << 1) - p2.a - (p2.a << 2);
  const s64 nA = WIDE_TERM(u0, A), nB = WIDE_TERM(u1, B), nC = WIDE_TERM(u2, C);
  const s64 nCl = WIDE_TERM(u0, Cl), nBl = WIDE_TERM(u1, Bl), nAl = WIDE_TERM(u2, Al);
#undef WIDE_TERM
  const s64 b = nB << 1, bl = nBl << 1;
  const s64 s = b + nC, sl = bl + nCl;
  const s64 Nh = nA + s + (s << 1), Nl = nAl - sl - (sl << 1);
  const bool bad = w_max(p0.x, w_max(p1.x, p2.x)) >= WIDE_X_BAD;
  const int x = z - y + 63;
  hi = w_fma(wide_quot(Nh, H, x, bad), 1.0 / 6.0, c);
  lo = w_fma(wide_quot(Nl, L, x, bad), 1.0 / 6.0, c);
}

// Both face values of the middle zone of a..e.
WIDE_FN void weno5_wide_pair(double a, double b, double c, double d, double e, double &lo,
                             double &hi) {
  const WideDiff f0 = wide_diff(b - a), f1 = wide_diff(c - b), f2 = wide_diff(d - c),
                 f3 = wide_diff(e - d);
  const WidePair p0 = wide_pair(f0, f1), p1 = wide_pair(f1, f2), p2 = wide_pair(f2, f3);
  weno5_wide(c, p0, p1, p2, wide_q_low(p0, wide_D13(p0)), wide_q_mid(p1, wide_D13(p1)),
             wide_q_high(p2, wide_D13(p2)), lo, hi);
}

}  // namespace grmhd
