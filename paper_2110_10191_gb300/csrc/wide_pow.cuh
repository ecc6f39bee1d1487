// wide_pow.cuh -- powers of Wide numbers (wide_num.cuh): log2 and 2^y.
//
// A power is 2^(a log2 x) with the logarithm and the exponent in fixed point of 55
// bits after the point: its relative error is 2^-55 and that of the
// product, where exp(a ln x) in doubles starts from a logarithm rounded to 2^-53 of its
// own size, up to 2^-49 for densities of 1e-7.
//
// Both reduce by a table of 64 entries over one octave and sum a Taylor series:
// log2 x = e + log2(1/r) + log2(1 + t) with r the 10-bit reciprocal of the interval's
// middle, so that t = m r - 1 is exact and below 2^-6.9 (eight terms, 2^-64), and
// 2^y = 2^n 2^(i/64) e^g with g below 2^-6.5 (seven, 2^-67).  Terms need fewer bits
// the higher they are: four of the logarithm's and four of the exponential's are
// taken in 32 bits.  About 150 issue cycles each, where log() and exp() take some
// 25 FP64 instructions of 76 cycles.
#pragma once

#include "wide_num.cuh"

namespace grmhd {

// 1024 / (1 + (i + 1/2)/64) rounded; log2 of 1024 over that, in 2^-55; 2^(i/64) in 2^-62
#define WIDE_POW_R \
    1016, 1001, 986, 971, 957, 943, 930, 917, 904, 892, 880, 868, 857, 846, 835, 824, \
    814, 804, 794, 785, 776, 767, 758, 749, 741, 732, 724, 716, 708, 701, 694, 686, \
    679, 672, 665, 659, 652, 646, 639, 633, 627, 621, 615, 610, 604, 599, 593, 588, \
    583, 577, 572, 567, 563, 558, 553, 548, 544, 539, 535, 531, 526, 522, 518, 514
#define WIDE_POW_L \
    0x172c7ba20f732ull, 0x431ee113bc5e5ull, 0x6fbb24546ab0cull, 0x9d067ab503625ull, \
    0xc7ef8e5477535ull, 0xf37a8616cfbaaull, 0x11c7e77dde33dcull, 0x146163957af02eull, \
    0x17046031c79f85ull, 0x197c1cb13c7ec1ull, 0x1bfc67a7fff4ccull, 0x1e857d3d361368ull, \
    0x20e06a4527ae49ull, 0x2343214bace941ull, 0x25add682a4649full, 0x2820c02f87d945ull, \
    0x2a61fa11e53f4eull, 0x2caa569330c4efull, 0x2efa036cdf7a6dull, 0x3114ed6fca938bull, \
    0x33360e552d8d65ull, 0x355d8b3b5b5b7cull, 0x378b8a9124a997ull, 0x39c03425ebb1a2ull, \
    0x3bbbd9f0e18983ull, 0x3dfd8c36023f0bull, 0x40050ccaf800cbull, 0x42125319ae3bbfull, \
    0x442580577b9367ull, 0x45fb3a5557f5c8ull, 0x47d5ab27b66a34ull, 0x49f9c8203f3797ull, \
    0x4bdea65fed4a97ull, 0x4dc88aedc1d1efull, 0x4fb790ba231e12ull, 0x5164091eb338f0ull, \
    0x535ce0373108b2ull, 0x5511edc9990e6bull, 0x5714fbe38b7b5eull, 0x58d2f876ac62cdull, \
    0x5a95346999d894ull, 0x5c5bc4a5ad539bull, 0x5e26beb02dc3eaull, 0x5fa8a8bb65f339ull, \
    0x617bf418b195b3ull, 0x6304ecde473c00ull, 0x64e0d828428580ull, 0x667122f8818f21ull, \
    0x6804d8e6620e93ull, 0x69ede538b7ec31ull, 0x6b8956067c08b3ull, 0x6d286396c81023ull, \
    0x6e771342e2e942ull, 0x701ccaf87a7faeull, 0x71c64e6d762159ull, 0x7373af48dce653ull, \
    0x74ce04829b7675ull, 0x7682885519a647ull, 0x77e2ab8391bd5aull, 0x7945733a7da824ull, \
    0x7b04b3dae5e976ull, 0x7c6d9388af5e0full, 0x7dd939dd0ad09eull, 0x7f47b1dc942a9cull
#define WIDE_POW_E \
    0x4000000000000000ull, 0x40b268f9de0183baull, 0x4166c34c5615d0ecull, 0x421d1461d66f2023ull, \
    0x42d561b3e6243d8aull, 0x438fb0cb4f468808ull, 0x444c0740496d4294ull, 0x450a6abaa4b77ecdull, \
    0x45cae0f1f545eb73ull, 0x468d6fadbf2dd4f3ull, 0x47521cc5a2e6a9e0ull, 0x4818ee218a3358eeull, \
    0x48e1e9b9d588e19bull, 0x49ad159789f37496ull, 0x4a7a77d47f7b84b1ull, 0x4b4a169b900c2d00ull, \
    0x4c1bf828c6dc54b8ull, 0x4cf022c9905bfd32ull, 0x4dc69cdceaa72a9cull, 0x4e9f6cd3967fdba8ull, \
    0x4f7a993048d088d7ull, 0x50582887dcb8a7e1ull, 0x513821818624b40cull, 0x521a8ad704f3404full, \
    0x52ff6b54d8a89c75ull, 0x53e6c9da74b29ab5ull, 0x54d0ad5a753e077cull, 0x55bd1cdad49f699cull, \
    0x56ac1f752150a563ull, 0x579dbc56b48521baull, 0x5891fac0e95612c8ull, 0x5988e20954889245ull, \
    0x5a827999fcef3242ull, 0x5b7ec8f19468bbc9ull, 0x5c7dd7a3b17dcf75ull, 0x5d7fad59099f22feull, \
    0x5e8451cfac061b5full, 0x5f8bccdb3d398841ull, 0x6096266533384a2bull, 0x61a3666d124bb204ull, \
    0x62b39508aa836d6full, 0x63c6ba6455dcd8aeull, 0x64dcdec3371793d1ull, 0x65f60a7f79393e2eull, \
    0x6712460a8fc24072ull, 0x683199ed779592caull, 0x69540ec8f895722dull, 0x6a79ad55e7f6fd10ull, \
    0x6ba27e656b4eb57aull, 0x6cce8ae13c57ebdbull, 0x6dfddbcbed791babull, 0x6f307a412f074892ull, \
    0x70666f76154a7089ull, 0x719fc4b95f452d29ull, 0x72dc8373be41a454ull, 0x741cb5281e25ee34ull, \
    0x75606373ee921c97ull, 0x76a7980f6cca15c2ull, 0x77f25ccdee6d7ae6ull, 0x7940bb9e2cffd89dull, \
    0x7a92be8a92436616ull, 0x7be86fb985689ddcull, 0x7d41d96db915019dull, 0x7e9f06067a4360baull
struct PowTables {
  u64 l[64], e[64];
  u32 r[64];
};
#ifdef __CUDACC__
static __device__ const PowTables w_pow_dev = {{WIDE_POW_L}, {WIDE_POW_E}, {WIDE_POW_R}};
#endif
static const PowTables w_pow_host = {{WIDE_POW_L}, {WIDE_POW_E}, {WIDE_POW_R}};

WIDE_FN u32 w_pow_r(u32 i) {
#ifdef __CUDA_ARCH__
  return __ldg(w_pow_dev.r + i);
#else
  return w_pow_host.r[i];
#endif
}
WIDE_FN u64 w_pow_l(u32 i) {
#ifdef __CUDA_ARCH__
  return __ldg(w_pow_dev.l + i);
#else
  return w_pow_host.l[i];
#endif
}
WIDE_FN u64 w_pow_e(u32 i) {
#ifdef __CUDA_ARCH__
  return __ldg(w_pow_dev.e + i);
#else
  return w_pow_host.e[i];
#endif
}
WIDE_FN u32 w_umulhi(u32 a, u32 b) { return w_hi(w_mul(a, b)); }

// positive, finite and within 2^-r .. 2^r
WIDE_FN bool w_within(double d, int r) {
  return (w_hi(w_bits(d)) >> 20) - (u32)(1023 - r) < (u32)(2 * r);
}

constexpr int LOG_BITS = 55;

// log2 a in 2^-55 for a positive normalised a below 2^250 and above 2^-250
WIDE_FN s64 w_log2(const Wide &a) {
  const u32 i = (w_hi(a.m) >> 24) & 63, r = w_pow_r(i);
  const s64 T = (s64)((w_mul(w_hi(a.m), r) << 22) + (w_mul(w_lo(a.m), r) >> 10) - (1ull << 62));
  const s64 s = w_sign(T);
  const u64 t = w_abs(T, s);  // |t| in 2^-62, below 2^55.1
  const u64 c = ~(u64)s;      // the series alternates for t > 0
  const u32 c32 = (u32)c, t30 = (u32)(t >> 30);
  // log2(e)/n, n = 8 .. 5 in 2^-32, then 4 .. 1 in 2^-62
  u32 q = 885189717u + ((w_umulhi(t30, 774541002u) ^ c32) - c32);
  q = 1032721336u + ((w_umulhi(t30, q) ^ c32) - c32);
  q = 1239265604u + ((w_umulhi(t30, q) ^ c32) - c32);
  u64 p = 0x171547652b82fe17ull + (((w_mul((u32)(t >> 24), q) >> 8) ^ c) - c);
  p = 0x1ec709dc3a03fd75ull + ((w_mulhi63(t << 2, p) ^ c) - c);
  p = 0x2e2a8eca5705fc2full + ((w_mulhi63(t << 2, p) ^ c) - c);
  p = 0x5c551d94ae0bf85eull + ((w_mulhi63(t << 2, p) ^ c) - c);
  return ((s64)(a.x + 62) << LOG_BITS) + (s64)w_pow_l(i) +
         w_signed(w_mulhi63(t << 7, p) >> 12, s);
}
// the logarithm as a normalised number, for its product with an exponent
WIDE_FN Wide w_log_num(s64 l) {
  Wide r;
  r.s = (int)(l >> 63);
  r.m = w_abs(l, (s64)r.s);
  r.x = -LOG_BITS;
  return norm(r);
}

// 2^y for |y| below 2^7 and y.m in [2^60, 2^62), a product of normalised numbers (or
// below 2^8 and y.m in [2^61, 2^62)); 0 for a y beyond that
WIDE_FN Wide w_exp2(const Wide &y) {
  const int sh = -LOG_BITS + 1 - y.x;
  const u64 q = w_shr(y.m << 1, w_max(sh, 0));
  const s64 Y = w_signed(q, (s64)y.s);
  const u64 f = (u64)Y & ((1ull << LOG_BITS) - 1);
  const u64 g = w_mulhi63((f & ((1ull << 49) - 1)) << 13, 0x58b90bfbe8e7bcd6ull);  // in 2^-67
  const u32 g32 = (u32)(g >> 35);
  // 1/n!, n = 7 .. 4 in 2^-36, then 3 .. 1 in 2^-62
  u32 h = 95443718u + w_umulhi(g32, 13634817u);
  h = 572662306u + w_umulhi(g32, h);
  h = 2863311531u + w_umulhi(g32, h);
  u64 p = 0xaaaaaaaaaaaaaabull + (w_mul((u32)(g >> 29), h) >> 12);
  p = 0x2000000000000000ull + w_mulhi63(g >> 3, p);
  p = 0x4000000000000000ull + w_mulhi63(g >> 3, p);
  const u64 e1 = w_mulhi63(g << 2, p);  // e^g - 1 in 2^-67
  const u64 t = w_pow_e((u32)(f >> 49));
  Wide r;
  r.m = t + (w_mulhi63(e1 << 2, t) >> 5);
  r.s = 0;
  r.x = (sh < 0) ? -1000 : (int)(Y >> LOG_BITS) - 62;
  if (sh < 0) r.m = 0;
  return r;
}

// The electrons' share of the heating in the model of Kawazura et al. (GRMHD_ELEC_KAWAZURA
// in grmhd.h), from rho, log2 rho (ls), u, kappa_e, all positive and normal, and any
// finite b^2:
// 1/(1 + 35/(1 + X)) = (1 + X)/(36 + X), X = (beta/15)^-1.4 exp(-0.1 T_e/T_p)
// ige: 1/(gamma_e - 1).
WIDE_FN Wide wide_kawazura(double game, double gamp, double ige, double rho, const Wide &ls,
                           double u, double kel, double bsq) {
  const Wide te = norm(wide_pos(kel) * w_exp2(ls * wide_pos(game - 1.0)));
  const Wide tr = norm(te * wide_pos(rho));                           // rho T_e
  Wide d = norm(norm(w_sum<1>(wide_pos(u), -(tr * wide_pos(ige)))));  // u_p
  d.s = 0;
  d = norm(d * wide_pos(gamp - 1.0));  // rho T_p
  constexpr s64 CLAMP = 0x213822cbd80c4db8ll, L15 = 0x1f414fdb498225all;  // log2 of 1e20 and of 15
  s64 lb = CLAMP;
  if ((s64)w_bits(bsq) > 0) {
    Wide beta = norm(d * w_rcp(norm(norm(wide(bsq)))));
    beta.x = w_min(w_max(beta.x + 1, -262), 138);
    lb = w_log2(beta);
    lb = lb < -CLAMP ? -CLAMP : lb > CLAMP ? CLAMP : lb;
  }
  const Wide t1 = w_log_num(lb - L15) * wide_pos(1.4);
  const Wide t2 = norm(tr * w_rcp(d)) * wide_pos(0.14426950408889634);  // log2(e)/10
  Wide y = norm(w_sum<1>(-t1, -t2));
  y.m >>= 1;
  y.x += 1;
  Wide X = w_exp2(y);
  if (d.m == 0) X.m = 0, X.x = -1000;  // no proton energy
  return norm(w_sum<1>(wide_pos(1.0), X) * w_rcp(norm(w_sum<1>(wide_pos(36.0), X))));
}

}  // namespace grmhd
