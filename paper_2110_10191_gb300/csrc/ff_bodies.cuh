// ff_bodies.cuh -- per-thread bodies of the float-float modes: the flux stage of
// GRMHD_PREC_FF (reconstruction, fluid states, signal speeds, local Lax-Friedrichs
// flux) and the source pass of the update of GRMHD_PREC_FF and
// GRMHD_PREC_MIXED_FF (U(P), geometric source), in float-float arithmetic (ff.cuh,
// about 48 significant bits) on the FP32 pipe; what is stored and the rest of the
// step as in the FP64 mode.  Same formulas as the FP64 mode's, with the energy
// flux and energy density formed without the rest-mass cancellation as in the
// FP32 bodies (grmhd_f32.cuh), since the 5 bits the float pair lacks would
// otherwise be lost 1e3-fold at rho >> u, and with every zone or face computed in
// units scaled by its density (FFScale).
//
// Data: the stage input split once per stage into high and low float words
// ([2][8][ntot]: all high words, then all low words), the face values in the
// same split layout, and a split copy of the geometry ([2][NLOC][G_NCOMP][n2d]).
#pragma once

#include "ff.cuh"
#include "grmhd_dev.cuh"
#include "step_bodies.cuh"

namespace grmhd {

__device__ __forceinline__ ff ff_load(const float *__restrict__ hi, long long lo_off, long long i) {
  ff r;
  r.hi = __ldg(hi + i);
  r.lo = __ldg(hi + lo_off + i);
  return r;
}

__device__ __forceinline__ void ff_store(float *hi, long long lo_off, long long i, ff v) {
  hi[i] = v.hi;
  hi[lo_off + i] = v.lo;
}

// Per-zone (per-face) scale.  Ideal MHD is invariant under rho, u, p, b^2 ->
// s (rho, u, p, b^2) with B -> sqrt(s) B and the velocities unchanged, so the
// float-float bodies work in units where the density is about 1: s = 4^m
// (an exact power of two whose square root 2^m is exact too) from the
// density; the hydrodynamic densities, fluxes and sources scale by s, the
// field and its fluxes by 2^m.  Without it the float exponent range
// (1e-38..3e38) cuts into floor-density atmospheres, where products such as
// (Q.B)^2 fall below 1e-38.
struct FFScale {
  float is, irs;  // 1/s, 1/sqrt(s): into the scaled units
  double s, rs;   // s, sqrt(s): back, applied in FP64
  int m;          // sqrt(s) = 2^m: back, on a double's exponent (d_scale)
};

__device__ __forceinline__ FFScale ff_scale_for(float rho) {
  int m = 0;
  if (rho > 0.0f) {
    m = ilogbf(rho) >> 1;  // floor of half the binary exponent
    m = max(-60, min(60, m));
  }
  FFScale c;
  c.is = ldexpf(1.0f, -2 * m);
  c.irs = ldexpf(1.0f, -m);
  c.s = ldexp(1.0, 2 * m);
  c.rs = ldexp(1.0, m);
  c.m = m;
  return c;
}

// a primitive vector into the scaled units (exact)
__device__ __forceinline__ void ff_scale_prims(ff P[NV], const FFScale &c) {
  P[RHO] = ff_ldexp(P[RHO], c.is);
  P[UU] = ff_ldexp(P[UU], c.is);
  P[B1] = ff_ldexp(P[B1], c.irs);
  P[B2] = ff_ldexp(P[B2], c.irs);
  P[B3] = ff_ldexp(P[B3], c.irs);
}

// one value split into its two words ([2][n]); values beyond the float
// range (inverse-metric components on the polar axis, which no flux reads)
// are clamped to +-FLT_MAX
__device__ __forceinline__ void to_ff_body(const double *__restrict__ src, float *__restrict__ dst,
                                           long long n, long long t) {
  if (t >= n) return;
  const double x = src[t];
  ff v;
  if ((w_hi(w_bits(x)) & 0x7fffffffu) >= (1151u << 20) && fabs(x) > 3.4028234663852886e38) {
    v.hi = (x > 0.0) ? 3.4028234663852886e38f : -3.4028234663852886e38f;
    v.lo = 0.0f;
  } else {
    v = ff_from_bits(x);
  }
  dst[t] = v.hi;
  dst[n + t] = v.lo;
}

// ---------------------------------------------------------------------------
// Reconstruction
// ---------------------------------------------------------------------------
// MC limited slope of x1 with neighbours x0, x2 (the FP64 body's decisions
// taken on the float-float differences)
__device__ __forceinline__ ff mc_slope_ff(ff x0, ff x1, ff x2) {
  const ff dm = ff_sub(x1, x0), dp = ff_sub(x2, x1);
  if (!((dm.hi > 0.0f && dp.hi > 0.0f) || (dm.hi < 0.0f && dp.hi < 0.0f))) return ff_f(0.0f);
  const ff dc = ff_ldexp(ff_add(dm, dp), 0.5f);
  const ff m = ff_min(ff_min(ff_abs(ff_ldexp(dm, 2.0f)), ff_abs(dc)), ff_abs(ff_ldexp(dp, 2.0f)));
  return (dc.hi > 0.0f) ? m : ff_neg(m);
}

// Both WENO5 face values of the middle zone of a..e: the FP64 body's
// first/second-difference form, with the weights d_k/(eps + beta_k)^2
// normalised by the power of two m below the smallest (eps + beta): r_k = m / e_k
// in (0, 1], so no product leaves the float exponent range (eps = 1e-26 makes
// e_k^2 as small as 1e-50); a weight that underflows is negligible next to the
// dominant one, which is above 1/4.
__device__ __forceinline__ void weno5_pair_ff(ff a, ff b, ff c, ff d, ff e, ff &lo, ff &hi) {
  const ff dm2 = ff_sub(b, a), dm1 = ff_sub(c, b), dp1 = ff_sub(d, c), dp2 = ff_sub(e, d);
  const ff D0 = ff_sub(dm1, dm2), D1 = ff_sub(dp1, dm1), D2 = ff_sub(dp2, dp1);
  const ff s0 = ff_add(D0, ff_ldexp(dm1, 2.0f));
  const ff s1 = ff_add(dm1, dp1);
  const ff s2 = ff_sub(D2, ff_ldexp(dp1, 2.0f));
  // 12 (eps + beta_k) = 12 eps + 13 D_k^2 + 3 s_k^2; 12 eps = 1.2e-25 split
  // into its float words (high 0x16148d85, low 0x89c7ce7b: the double
  // constant to 2e-41)
  ff eps12;
  eps12.hi = __int_as_float(0x16148d85);
  eps12.lo = __int_as_float((int)0x89c7ce7bu);
  const ff e0 = ff_add(ff_add(ff_mul_f(ff_sqr(D0), 13.0f), ff_mul_f(ff_sqr(s0), 3.0f)), eps12);
  const ff e1 = ff_add(ff_add(ff_mul_f(ff_sqr(D1), 13.0f), ff_mul_f(ff_sqr(s1), 3.0f)), eps12);
  const ff e2 = ff_add(ff_add(ff_mul_f(ff_sqr(D2), 13.0f), ff_mul_f(ff_sqr(s2), 3.0f)), eps12);
  const float m = __int_as_float(__float_as_int(fminf(fminf(e0.hi, e1.hi), e2.hi)) & 0x7f800000);
  const ff r0 = ff_ldexp(ff_rcp(e0), m), r1 = ff_ldexp(ff_rcp(e1), m), r2 = ff_ldexp(ff_rcp(e2), m);
  const ff w0 = ff_sqr(r0), w1 = ff_mul_f(ff_sqr(r1), 6.0f), w2 = ff_sqr(r2);
  const ff w2x3 = ff_mul_f(w2, 3.0f), w0x3 = ff_mul_f(w0, 3.0f);
  const ff m3 = ff_mul_f(dm1, 3.0f), p3 = ff_mul_f(dp1, 3.0f);
  // high face: linear weights 1 : 6 : 3 on stencils 0, 1, 2
  const ff nh = ff_add(ff_add(ff_mul(w0, ff_add(ff_ldexp(D0, 2.0f), m3)),
                              ff_mul(w1, ff_add(dm1, ff_ldexp(dp1, 2.0f)))),
                       ff_mul(w2x3, ff_sub(p3, D2)));
  const ff H = ff_mul_f(ff_add(ff_add(w0, w1), w2x3), 6.0f);
  // low face: the mirrored stencils (2, 1, 0) with the same linear weights
  const ff nl = ff_sub(ff_sub(ff_mul(w2, ff_sub(ff_ldexp(D2, 2.0f), p3)),
                              ff_mul(w1, ff_add(dp1, ff_ldexp(dm1, 2.0f)))),
                       ff_mul(w0x3, ff_add(m3, D0)));
  const ff L = ff_mul_f(ff_add(ff_add(w2, w1), w0x3), 6.0f);
  hi = ff_add(c, ff_div(nh, H));
  lo = ff_add(c, ff_div(nl, L));
}

// Zone-centric reconstruction along DIR in float-float: Pff is the split
// stage input ([2][8][ntot]), Lf/Rf the split low/high face values.
template <int DIR, int RECON>
__device__ __forceinline__ void recon_ff_body(const StepArgs &A, const float *__restrict__ Pff,
                                              float *__restrict__ Lf, float *__restrict__ Rf,
                                              long long t) {
  const Dims &D = A.D;
  const int e0 = D.n[0] + 2, e1 = D.n[1] + 2;
  if (t >= n_recon(D, A.flat3)) return;
  const Idx3 q3 = unflatten(t, e0, e1);
  const int i = NG - 1 + q3.i, j = NG - 1 + q3.j, k = (A.flat3 ? NG : NG - 1) + q3.k;
  const long long c = zid(D, i, j, k);
  const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
  const long long half = (long long)NV * D.ntot;
#pragma unroll 1
  for (int v = 0; v < NV; v++) {
    const long long o = v * D.ntot + c;
    ff lo, hi;
    if (RECON == 1) {
      weno5_pair_ff(ff_load(Pff, half, o - 2 * st), ff_load(Pff, half, o - st), ff_load(Pff, half, o),
                    ff_load(Pff, half, o + st), ff_load(Pff, half, o + 2 * st), lo, hi);
    } else {
      const ff x1 = ff_load(Pff, half, o);
      const ff h = ff_ldexp(mc_slope_ff(ff_load(Pff, half, o - st), x1, ff_load(Pff, half, o + st)), 0.5f);
      lo = ff_sub(x1, h);
      hi = ff_add(x1, h);
    }
    ff_store(Lf, half, o, lo);
    ff_store(Rf, half, o, hi);
  }
}

// ---------------------------------------------------------------------------
// Face fluxes
// ---------------------------------------------------------------------------
struct GeoFF {
  ff gcov[10], gcon[10], gdet, alpha, ialpha, omalpha, igdet;
};

// geometry of one location from the split copy ([2][NLOC][G_NCOMP][n2d];
// g points at this location's components, lo_off = NLOC G_NCOMP n2d)
__device__ __forceinline__ void load_geo_ff(const float *__restrict__ g, long long lo_off, long long n2d,
                                            long long ij, GeoFF &G) {
#pragma unroll
  for (int q = 0; q < 10; q++) G.gcov[q] = ff_load(g, lo_off, (G_GCOV + q) * n2d + ij);
#pragma unroll
  for (int q = 0; q < 10; q++) G.gcon[q] = ff_load(g, lo_off, (G_GCON + q) * n2d + ij);
  G.gdet = ff_load(g, lo_off, G_GDET * n2d + ij);
  G.alpha = ff_load(g, lo_off, G_ALPHA * n2d + ij);
  G.ialpha = ff_load(g, lo_off, G_IALPHA * n2d + ij);
  G.omalpha = ff_load(g, lo_off, G_OMALPHA * n2d + ij);
  G.igdet = ff_load(g, lo_off, G_IGDET * n2d + ij);
}

// Fluid state as fluid_state (grmhd_dev.cuh), plus opu_t = 1 + u_t formed
// as (1 - alpha) - alpha (gamma - 1) + g_tj utilde^j, gamma - 1 = q^2/(1 + gamma).
struct FStateFF {
  ff ucon[4], ucov[4], bcon[4], bcov[4], bsq, opu_t;
};

__device__ __forceinline__ ff dot3(ff a0, ff b0, ff a1, ff b1, ff a2, ff b2) {
  return ff_add(ff_add(ff_mul(a0, b0), ff_mul(a1, b1)), ff_mul(a2, b2));
}

__device__ __forceinline__ void fluid_state_ff(const ff P[NV], const GeoFF &G, FStateFF &s) {
  const ff v1 = P[U1], v2 = P[U2], v3 = P[U3];
  const ff l1 = dot3(G.gcov[SY(1, 1)], v1, G.gcov[SY(1, 2)], v2, G.gcov[SY(1, 3)], v3);
  const ff l2 = dot3(G.gcov[SY(1, 2)], v1, G.gcov[SY(2, 2)], v2, G.gcov[SY(2, 3)], v3);
  const ff l3 = dot3(G.gcov[SY(1, 3)], v1, G.gcov[SY(2, 3)], v2, G.gcov[SY(3, 3)], v3);
  const ff qsq = dot3(l1, v1, l2, v2, l3, v3);
  const ff g2 = ff_add_f(qsq, 1.0f);
  const ff rg = ff_rsqrt(g2);
  const ff gam = ff_mul(g2, rg);
  const ff ga = ff_mul(gam, G.alpha);
  const ff sh = dot3(G.gcov[SY(0, 1)], v1, G.gcov[SY(0, 2)], v2, G.gcov[SY(0, 3)], v3);
  s.opu_t = ff_add(ff_sub(G.omalpha, ff_mul(ff_mul(G.alpha, qsq), ff_rcp(ff_add_f(gam, 1.0f)))), sh);
  s.ucon[0] = ff_mul(gam, G.ialpha);
  s.ucon[1] = ff_sub(v1, ff_mul(ga, G.gcon[SY(0, 1)]));
  s.ucon[2] = ff_sub(v2, ff_mul(ga, G.gcon[SY(0, 2)]));
  s.ucon[3] = ff_sub(v3, ff_mul(ga, G.gcon[SY(0, 3)]));
  s.ucov[0] = ff_sub(sh, ga);
  s.ucov[1] = l1;
  s.ucov[2] = l2;
  s.ucov[3] = l3;
  const ff bt = dot3(P[B1], l1, P[B2], l2, P[B3], l3);
  const ff iut = ff_mul(G.alpha, rg);  // 1/u^t
  s.bcon[0] = bt;
  s.bcon[1] = ff_mul(ff_add(P[B1], ff_mul(bt, s.ucon[1])), iut);
  s.bcon[2] = ff_mul(ff_add(P[B2], ff_mul(bt, s.ucon[2])), iut);
  s.bcon[3] = ff_mul(ff_add(P[B3], ff_mul(bt, s.ucon[3])), iut);
#pragma unroll
  for (int m = 0; m < 4; m++) {
    ff a = ff_f(0.0f);
#pragma unroll
    for (int n = 0; n < 4; n++) a = ff_add(a, ff_mul(G.gcov[SY(m, n)], s.bcon[n]));
    s.bcov[m] = a;
  }
  s.bsq = ff_add(ff_add(ff_mul(s.bcon[0], s.bcov[0]), ff_mul(s.bcon[1], s.bcov[1])),
                 ff_add(ff_mul(s.bcon[2], s.bcov[2]), ff_mul(s.bcon[3], s.bcov[3])));
}

// acc += F^dir + coef U without the sqrt(-g) factor (flux_cons_acc), the
// energy row as rho uc (1 + u_t) + (w - rho) uc u_t - bc b_t + coef pt
__device__ __forceinline__ void flux_cons_acc_ff(const ff P[NV], const FStateFF &s, ff gm1,
                                                 int dir, ff coef, ff acc[NV]) {
  const ff pg = ff_mul(P[UU], gm1);
  const ff w = ff_add(ff_add(P[RHO], P[UU]), ff_add(pg, s.bsq));
  const ff pt = ff_add(pg, ff_ldexp(s.bsq, 0.5f));
  const ff uc = ff_add(s.ucon[dir], ff_mul(coef, s.ucon[0]));
  const ff bc = ff_add(s.bcon[dir], ff_mul(coef, s.bcon[0]));
  const ff wuc = ff_mul(w, uc);
  ff T[4];
#pragma unroll
  for (int nu = 0; nu < 4; nu++) T[nu] = ff_sub(ff_mul(wuc, s.ucov[nu]), ff_mul(bc, s.bcov[nu]));
  T[dir] = ff_add(T[dir], pt);
  const ff mf = ff_mul(P[RHO], uc);
  acc[RHO] = ff_add(acc[RHO], mf);
  const ff en = ff_add(ff_mul(mf, s.opu_t),
                       ff_sub(ff_mul(ff_mul(ff_sub(w, P[RHO]), uc), s.ucov[0]), ff_mul(bc, s.bcov[0])));
  acc[UU] = ff_add(acc[UU], ff_add(en, ff_mul(coef, pt)));
  acc[U1] = ff_add(acc[U1], T[1]);
  acc[U2] = ff_add(acc[U2], T[2]);
  acc[U3] = ff_add(acc[U3], T[3]);
  acc[B1] = ff_add(acc[B1], ff_sub(ff_mul(s.bcon[1], uc), ff_mul(bc, s.ucon[1])));
  acc[B2] = ff_add(acc[B2], ff_sub(ff_mul(s.bcon[2], uc), ff_mul(bc, s.ucon[2])));
  acc[B3] = ff_add(acc[B3], ff_sub(ff_mul(s.bcon[3], uc), ff_mul(bc, s.ucon[3])));
}

// fast magnetosonic speeds along dir (the quadratic of mhd_cmax)
// gam: the adiabatic index, ggm1 = gam (gam - 1), both float-float
__device__ __forceinline__ void mhd_vchar_ff(const ff P[NV], const FStateFF &s, const GeoFF &G,
                                             ff gam, ff ggm1, int dir, ff &vmax, ff &vmin) {
  // cs2 + va2 - cs2 va2 = (gamma (gamma - 1) u + b^2) / (b^2 + e_f) exactly
  const ff ef = ff_add(P[RHO], ff_mul(P[UU], gam));
  const ff ee = ff_add(s.bsq, ef);
  const ff cms2 = ff_mul(ff_add(ff_mul(P[UU], ggm1), s.bsq), ff_rcp(ee));
  const ff Asq = G.gcon[SY(dir, dir)];
  const ff Bsq = G.gcon[SY(0, 0)];
  const ff AB = G.gcon[SY(0, dir)];
  const ff Au = s.ucon[dir];
  const ff Bu = s.ucon[0];
  const ff AuBu = ff_mul(Au, Bu);
  const ff qa = ff_sub(ff_sqr(Bu), ff_mul(ff_add(Bsq, ff_sqr(Bu)), cms2));
  const ff qb = ff_mul_f(ff_sub(AuBu, ff_mul(ff_add(AB, AuBu), cms2)), -2.0f);
  const ff qc = ff_sub(ff_sqr(Au), ff_mul(ff_add(Asq, ff_sqr(Au)), cms2));
  ff disc = ff_sub(ff_sqr(qb), ff_mul_f(ff_mul(qa, qc), 4.0f));
  disc = (disc.hi > 0.0f) ? ff_sqrt(disc) : ff_f(0.0f);
  const ff i2a = ff_ldexp(ff_rcp(qa), 0.5f);
  const ff v1 = ff_mul(ff_add(ff_neg(qb), disc), i2a);
  const ff v2 = ff_mul(ff_sub(ff_neg(qb), disc), i2a);
  vmax = ff_max(v1, v2);
  vmin = ff_min(v1, v2);
}

// One thread per face: split states Rf(c - st) (left) and Lf(c) (right),
// split geometry; the LLF flux stored in FP64.  Every thread of the block
// must call it (signal-speed block maximum).
template <int DIR>
__device__ __forceinline__ void face_ff_body(const StepArgs &A, const float *__restrict__ geomff,
                                             const float *__restrict__ Lf,
                                             const float *__restrict__ Rf, double *__restrict__ F,
                                             long long t) {
  const Dims &D = A.D;
  int lo[3], ext[3];
  face_box(D, DIR, A.flat3, lo, ext);
  const long long nface = (long long)ext[0] * ext[1] * ext[2];
  const bool active = t < nface;
  double ctop = 0.0;
  if (active) {
    const Idx3 q3 = unflatten(t, ext[0], ext[1]);
    const int i = lo[0] + q3.i, j = lo[1] + q3.j, k = lo[2] + q3.k;
    const long long c = zid(D, i, j, k);
    const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
    const long long half = (long long)NV * D.ntot;
    ff PL[NV], PR[NV];
#pragma unroll
    for (int v = 0; v < NV; v++) {
      PL[v] = ff_load(Rf, half, v * D.ntot + c - st);
      PR[v] = ff_load(Lf, half, v * D.ntot + c);
    }
    const int loc = (DIR == 0) ? LOC_FACE1 : (DIR == 1) ? LOC_FACE2 : LOC_CENT;
    GeoFF G;
    load_geo_ff(geomff + (long long)loc * G_NCOMP * D.n2d, (long long)NLOC * G_NCOMP * D.n2d, D.n2d,
                (long long)j * D.s[0] + i, G);
    const ff gam = {A.gam_ff[0], A.gam_ff[1]}, gm1 = {A.gm1_ff[0], A.gm1_ff[1]};
    const ff ggm1 = {A.ggm1_ff[0], A.ggm1_ff[1]};
    FStateFF sL, sR;
    const FFScale sc = ff_scale_for(PL[RHO].hi);
    ff_scale_prims(PL, sc);
    ff_scale_prims(PR, sc);
    fluid_state_ff(PL, G, sL);
    fluid_state_ff(PR, G, sR);
    ff vmaxL, vminL, vmaxR, vminR;
    mhd_vchar_ff(PL, sL, G, gam, ggm1, DIR + 1, vmaxL, vminL);
    mhd_vchar_ff(PR, sR, G, gam, ggm1, DIR + 1, vmaxR, vminR);
    const ff z = ff_f(0.0f);
    const ff cmax = ff_max(ff_max(z, vmaxL), vmaxR);
    const ff cmin = ff_max(ff_max(z, ff_neg(vminL)), ff_neg(vminR));
    const ff ct = ff_max(cmax, cmin);
    ff acc[NV];
#pragma unroll
    for (int v = 0; v < NV; v++) acc[v] = z;
    flux_cons_acc_ff(PL, sL, gm1, DIR + 1, ct, acc);
    flux_cons_acc_ff(PR, sR, gm1, DIR + 1, ff_neg(ct), acc);
    const ff hg = ff_ldexp(G.gdet, 0.5f);
#pragma unroll
    for (int v = 0; v < NV; v++)
      F[v * D.ntot + c] = ff_to(ff_mul(hg, acc[v])) * (v < B1 ? sc.s : sc.rs);
    if (A.elec_w) {  // the electron entropies' flux weights (rho scales with s)
      const ff wl = ff_mul(hg, ff_mul(PL[RHO], ff_add(sL.ucon[DIR + 1], ff_mul(ct, sL.ucon[0]))));
      const ff wr = ff_mul(hg, ff_mul(PR[RHO], ff_sub(sR.ucon[DIR + 1], ff_mul(ct, sR.ucon[0]))));
      A.elec_w[(2 * DIR) * D.ntot + c] = ff_to(wl) * sc.s;
      A.elec_w[(2 * DIR + 1) * D.ntot + c] = ff_to(wr) * sc.s;
    }
    bool interior = true;
#pragma unroll
    for (int e = 0; e < 3; e++) {
      if (e == DIR) continue;
      const int q = (e == 0) ? i : (e == 1) ? j : k;
      interior = interior && (q >= NG) && (q < D.n[e] + NG);
    }
    if (interior) ctop = ff_to(ct);
  }
  warp_block_max(ctop, &A.clk->ctop_bits[DIR]);
}

// ---------------------------------------------------------------------------
// The update's source pass in float-float
// ---------------------------------------------------------------------------
// sqrt(-g)-weighted conserved densities of a state (prim_flux with dir 0) but
// the field's,
// the energy density without the rest-mass cancellation:
// T^t_t + rho u^t = rho u^t (1 + u_t) + (w - rho) u^t u_t - b^t b_t + p_t
__device__ __forceinline__ void prim_cons_ff(const ff P[NV], const FStateFF &s, const GeoFF &G, ff gm1,
                                             ff U[B1]) {
  const ff pg = ff_mul(P[UU], gm1);
  const ff w = ff_add(ff_add(P[RHO], P[UU]), ff_add(pg, s.bsq));
  const ff pt = ff_add(pg, ff_ldexp(s.bsq, 0.5f));
  const ff ut = s.ucon[0], bt = s.bcon[0];
  const ff wu = ff_mul(w, ut);
  const ff mf = ff_mul(P[RHO], ut);
  U[RHO] = ff_mul(G.gdet, mf);
  const ff en = ff_add(ff_add(ff_mul(mf, s.opu_t), ff_mul(ff_mul(ff_sub(w, P[RHO]), ut), s.ucov[0])),
                       ff_sub(pt, ff_mul(bt, s.bcov[0])));
  U[UU] = ff_mul(G.gdet, en);
#pragma unroll
  for (int i = 1; i < 4; i++) U[UU + i] = ff_mul(G.gdet, ff_sub(ff_mul(wu, s.ucov[i]), ff_mul(bt, s.bcov[i])));
}

// S_nu = sqrt(-g) T^k_l Gamma^l_{nu k} (geo_source) from the split connection
__device__ __forceinline__ void geo_source_ff(const ff P[NV], const FStateFF &s, const GeoFF &G,
                                              const float *__restrict__ connff, long long lo_off,
                                              long long n2d, long long ij, ff gm1, ff S[4]) {
  const ff pg = ff_mul(P[UU], gm1);
  const ff w = ff_add(ff_add(P[RHO], P[UU]), ff_add(pg, s.bsq));
  const ff pt = ff_add(pg, ff_ldexp(s.bsq, 0.5f));
  ff T[4][4];
#pragma unroll
  for (int m = 0; m < 4; m++) {
    const ff wu = ff_mul(w, s.ucon[m]);
#pragma unroll
    for (int n = 0; n < 4; n++) T[m][n] = ff_sub(ff_mul(wu, s.ucov[n]), ff_mul(s.bcon[m], s.bcov[n]));
    T[m][m] = ff_add(T[m][m], pt);
  }
#pragma unroll
  for (int nu = 0; nu < 4; nu++) {
    ff acc = ff_f(0.0f);
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int l = 0; l < 4; l++)
        acc = ff_add(acc, ff_mul(T[k][l], ff_load(connff, lo_off, (l * 10 + SY(nu, k)) * n2d + ij)));
    S[nu] = ff_mul(acc, G.gdet);
  }
}

// source_body with U(P) and the source in float-float (one thread per zone, in
// units scaled by the zone's density); the field's part and what is stored are
// FP64.  Pff (may be null): the split stage input of the flux stage, which is P_s.
// (As one pass with a float-float inversion the update took 1.06 to 1.16 ms per
// launch on a 128^3 grid, bound by latency at 16 warps per SM; with the Wide
// inversion as a pass of its own, 0.79 ms for both.)
template <bool PRED>
__device__ __forceinline__ void source_ff_body(const StepArgs &A, const double *__restrict__ Ps,
                                               const float *__restrict__ Pff,
                                               double *__restrict__ Ucache,
                                               double *__restrict__ scratch, long long t) {
  const Dims &D = A.D;
  if (t >= n_update(D)) return;
  const Column q3 = column_of(t, (int)(t & 31), 32, D.n[0], D.n[1], D.n[2]);
  if (!q3.active) return;
  const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
  const long long c = zid(D, i, j, k), N = D.ntot;
  const long long ij = (long long)j * D.s[0] + i;
  GeoFF G;
  load_geo_ff(A.geomff, (long long)NLOC * G_NCOMP * D.n2d, D.n2d, ij, G);
  const ff gm1 = {A.gm1_ff[0], A.gm1_ff[1]};
  ff p[NV], S[4];
#pragma unroll
  for (int v = 0; v < NV; v++)
    p[v] = Pff ? ff_load(Pff, (long long)NV * N, v * N + c) : ff_from(__ldg(Ps + v * N + c));
  const FFScale sc = ff_scale_for(p[RHO].hi);
  ff_scale_prims(p, sc);
  FStateFF s;
  fluid_state_ff(p, G, s);
  if (PRED) {
    ff U[B1];
    prim_cons_ff(p, s, G, gm1, U);
    const double gd = __ldg(A.geom + (long long)G_GDET * D.n2d + ij);
#pragma unroll
    for (int v = 0; v < B1; v++) Ucache[v * N + c] = d_scale(ff_to_bits(U[v]), 2 * sc.m);
#pragma unroll
    for (int v = B1; v < NV; v++) Ucache[v * N + c] = gd * __ldg(Ps + v * N + c);
  }
  geo_source_ff(p, s, G, A.connff, (long long)C_NCOMP * D.n2d, D.n2d, ij, gm1, S);
#pragma unroll
  for (int n = 0; n < 4; n++) scratch[n * N + c] = d_scale(ff_to_bits(S[n]), 2 * sc.m);
  // the inversion's guess W = (rho + gamma u) gamma_L^2, to FP32
  const float lor = s.ucon[0].hi * G.alpha.hi;
  scratch[SCR_GUESS * N + c] =
      d_scale(f_to_double(fmaf(A.gam_ff[0], p[UU].hi, p[RHO].hi) * (lor * lor)), 2 * sc.m);
  if (A.elec) scratch[SCR_BSQ_S * N + c] = d_scale(ff_to_bits(s.bsq), 2 * sc.m);
}

}  // namespace grmhd
