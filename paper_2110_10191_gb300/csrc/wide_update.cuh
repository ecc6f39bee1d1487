// wide_update.cuh -- the conserved densities, the stress-energy tensor and the
// 1D_W inversion of one zone in Wide numbers (wide_num.cuh): the formulas of
// prim_flux (direction 0), geo_source and invert_1dw.
#pragma once

#include <math.h>

#include "wide_face.cuh"

namespace grmhd {

// Rows of a state, rounded to double: U(P) but its field part (WANT_U) and T^k_l.
// g2, bsq: the Lorentz factor squared and b^2.
template <bool BLK, bool WANT_U, class GeoFn>
WIDE_FN void wide_tensor(const double P[NV], const GeoFn &geo, double gm1, double U[NV],
                         double T[4][4], double &g2, double &bsq) {
  WideState s;
  wide_state<BLK>(P, geo, s);
  g2 = w_to_double(s.g2);
  bsq = w_to_double(s.bsq);
  const Wide rho = wide(P[RHO]), u = wide(P[UU]), pg = wide(gm1) * u;
  const Wide w = norm(w_sum<2>(rho, u, pg, s.bsq));
  const Wide pt = w_sum<1>(pg, w_scale(s.bsq, -1));
  Wide bcov[4];
#pragma unroll
  for (int n = 0; n < 4; n++) bcov[n] = norm(w_sum<1>(s.Bcov[n], s.bt * s.ucov[n])) * s.iut;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const Wide bk =
        k ? norm(w_sum<1>(wide(P[B1 - 1 + (k ? k : 1)]), s.bt * s.ucon[k])) * s.iut : s.bt;
    const Wide wu = norm(w * s.ucon[k]), nb = -norm(bk);
    const Wide gd = wide_pos(geo(G_GDET));
#pragma unroll
    for (int l = 0; l < 4; l++) {
      const Wide t = (k == l) ? w_sum<1>(wu * s.ucov[l], nb * bcov[l], pt)
                              : w_sum<0>(wu * s.ucov[l], nb * bcov[l]);
      T[k][l] = w_to_double(t);
      if (WANT_U && k == 0) {
        if (l == 0) {
          const Wide mf = rho * s.ucon[0];
          U[RHO] = w_to_double(mf * gd);
          U[UU] = w_to_double(w_sum<1>(t, mf) * gd);
        } else {
          U[UU + l] = w_to_double(t * gd);
        }
      }
    }
  }
}

// The 1D_W function f(W') and its derivative in FP32 (all quantities in units of a
// power of two near W)
struct InvF {
  float d, b, qt2, qb2, c, gf;  // D, B^2, Qt^2, (Q.B)^2, Q'.n + B^2, (gamma - 1)/gamma
};
WIDE_FN float inv_rcpf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}
WIDE_FN float inv_rsqrtf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}
// df/dW' from W, 1 - v^2, the Lorentz factor rs and b^2 = B^2 (1 - v^2) + (Q.B/W)^2.  With
// dv^2/dW = -2 (v^2 W + (Q.B/W)^2) / (W (B^2 + W)) the derivative of the formula below is
//   df = A (1 - 2 gf + gf r) + gf (1 - v^2) (1 - r),
// A = (W + b^2)/(W + B^2), r = D rs / W = rho / (rho + gamma u): no difference of large
// terms at any Lorentz factor or magnetisation (gamma <= 2), so that it has the relative
// accuracy of 1 - v^2.
WIDE_FN float inv_df(const InvF &q, float w, float omv, float rs, float b2) {
  const float r = q.d * rs * inv_rcpf(w), A = (w + b2) * inv_rcpf(w + q.b);
  return A * ((1.0f - 2.0f * q.gf) + q.gf * r) + q.gf * omv * (1.0f - r);
}
// v^2; f and df are meaningless for v^2 >= 1
WIDE_FN float inv_f32(const InvF &q, float wp, float &f, float &df) {
  const float w = wp + q.d, iw = inv_rcpf(w), ib = inv_rcpf(q.b + w);
  const float x2 = q.qb2 * iw * iw;
  const float vsq = (q.qt2 + x2 * (q.b + 2.0f * w)) * ib * ib;
  const float omv = 1.0f - vsq, rs = inv_rsqrtf(omv), sq = omv * rs, b2 = q.b * omv + x2;
  const float wmr = wp * omv - q.d * vsq * sq * inv_rcpf(1.0f + sq);
  f = q.c + wp - q.gf * wmr - 0.5f * b2;
  df = inv_df(q, w, omv, rs, b2);
  return vsq;
}

// The 1D_W inversion where nothing unusual happens: Newton steps in FP32 from the
// guess W until they are below 1e-5 (or twelve; an iterate beyond v^2 = 1 lies below the
// root and is replaced by the middle between it and the least W' above the root, or doubled
// while none is known: without the bracket Newton and doubling alternated for good
// at Lorentz factors above 8, and up to 88% of such states were left to FP64), then
// Newton steps whose function is taken in Wide numbers and whose derivative in FP32 of
// Wide values (each gains 20 bits or doubles the digits), until what f leaves is below
// 2^-INV_RESIDUAL of B^2 or of its largest term, about the noise of its own operations
// (1/(W (B^2 + W)) is good to 2^-57): a step's size says nothing where the derivative
// may be off.  The state comes from the pass that finds f so.  False, with nothing written, where the iteration of invert_1dw is needed for its answer or
// its failure code: input that is not finite, D <= 0, an iterate with
// v^2 > 1 - 1e-10, no convergence, u < 0.
//
// Worst relative errors of rho and u over 600 states each, unmagnetised to b^2 = 400 rho,
// u = 1e-6 to 1 rho, adiabatic indices 4/3 and 5/3, against the root in 113 bits, here and
// of the FP64 iteration: Lorentz factors 1 to 3, rho 5e-15 and 1e-13, u 2e-9 and 9e-8; 20 to
// 50, rho 1e-12 and 7e-11, u 5e-7 and 1e-5.  Three passes, 3.3 at 20 to 50; the update of
// a 96^3 grid takes 0.69 to 0.71 ms a cycle at Lorentz factors of 1.1 to 30 (3.18 at 30 with
// adiabatic index 5/3 when every zone there went on to FP64).
constexpr int INV_F32_MAXIT = 12, INV_WIDE_MAXIT = 8;
constexpr int INV_RESIDUAL = 56;

template <bool BLK, class GeoFn>
WIDE_FN bool wide_invert(const double U[NV], const GeoFn &geo, const GasK &K, double guess,
                         double P[NV], double &bsq_out, double &lorentz_out) {
#define GCOV(m, n) wide(geo(G_GCOV + SY(m, n)))
#define GDIA(m) wide_pos(geo(G_GCOV + SY(m, m)))
#define GCON(m, n) wide(geo(G_GCON + SY(m, n)))
  bool ok = true;
#pragma unroll
  for (int v = 0; v < NV; v++) ok = ok && w_finite(U[v]);
  const double igd = geo(G_IGDET);
  double b[3];
#pragma unroll
  for (int i = 0; i < 3; i++) b[i] = U[B1 + i] * igd;
  const Wide al = wide_pos(geo(G_ALPHA)), wigd = wide_pos(igd), aig = norm(al * wigd);
  const Wide n1 = al * wide(b[0]), n2 = al * wide(b[1]), n3 = al * wide(b[2]);  // normal-frame field
  const Wide urho = wide(U[RHO]);
  const Wide D = norm(urho * aig);
  ok = ok && D.s == 0 && D.m != 0;
  const Wide Q1 = norm(aig * wide(U[U1])), Q2 = norm(aig * wide(U[U2])), Q3 = norm(aig * wide(U[U3]));
  // c.Q with c_i = g^{ti}; Q'.n = (U_u - (1 - alpha) U_rho) / sqrt(-g) - alpha c.Q;
  // Qt^i = gamma^ij Q_j = g^ij Q_j + alpha^2 c^i c.Q
  const Wide c1 = GCON(0, 1), c3 = GCON(0, 3);
  Wide cQ, Qt1, Qt2, Qt3, Bsq;
  if (BLK) {
    cQ = norm(w_sum<0>(c1 * Q1, c3 * Q3));
  } else {
    cQ = norm(w_sum<1>(c1 * Q1, GCON(0, 2) * Q2, c3 * Q3));
  }
  const Wide acQ = norm(al * cQ), a2cQ = norm(al * acQ);
  const Wide Qpn = norm(w_sum<1>(
      norm(w_sum<1>(wide(U[UU]), -(wide(geo(G_OMALPHA)) * urho))) * wigd, -acQ));
  if (BLK) {
    const Wide g13 = GCON(1, 3), h13 = GCOV(1, 3);
    Qt1 = norm(w_sum<1>(GCON(1, 1) * Q1, g13 * Q3, c1 * a2cQ));
    Qt2 = norm(GCON(2, 2) * Q2);
    Qt3 = norm(w_sum<1>(g13 * Q1, GCON(3, 3) * Q3, c3 * a2cQ));
    Bsq = norm(w_sum<1>(n1 * norm(w_sum<0>(GDIA(1) * n1, h13 * n3)), n2 * norm(GDIA(2) * n2),
                        n3 * norm(w_sum<0>(h13 * n1, GDIA(3) * n3))));
  } else {
    const Wide g12 = GCON(1, 2), g13 = GCON(1, 3), g23 = GCON(2, 3);
    const Wide h12 = GCOV(1, 2), h13 = GCOV(1, 3), h23 = GCOV(2, 3);
    Qt1 = norm(w_sum<1>(GCON(1, 1) * Q1, g12 * Q2, g13 * Q3, c1 * a2cQ));
    Qt2 = norm(w_sum<1>(g12 * Q1, GCON(2, 2) * Q2, g23 * Q3, GCON(0, 2) * a2cQ));
    Qt3 = norm(w_sum<1>(g13 * Q1, g23 * Q2, GCON(3, 3) * Q3, c3 * a2cQ));
    Bsq = norm(w_sum<1>(n1 * norm(w_sum<1>(GDIA(1) * n1, h12 * n2, h13 * n3)),
                        n2 * norm(w_sum<1>(h12 * n1, GDIA(2) * n2, h23 * n3)),
                        n3 * norm(w_sum<1>(h13 * n1, h23 * n2, GDIA(3) * n3))));
  }
  const Wide Qtsq = norm(w_sum<1>(Qt1 * Q1, Qt2 * Q2, Qt3 * Q3));
  const Wide QdB = norm(w_sum<1>(Q1 * n1, Q2 * n2, Q3 * n3));
  ok = ok && w_finite(guess) && (Qtsq.s == 0 || Qtsq.m == 0) && (Bsq.s == 0 || Bsq.m == 0);

  // f = Q'.n + W' - gf (w - rho) + (1 + v^2) B^2/2 - (Q.B/W)^2/2 = C + W' - gf (w - rho) - b^2/2
  const Wide C = norm(w_sum<1>(Qpn, Bsq));

  // the guess, improved in FP32
  Wide Wp = norm(w_sum<1>(wide(guess), -D));
  const int e = -(int)((w_hi(w_bits(guess)) >> 20) & 0x7ff) + 1023;  // guess 2^e in [1, 2)
  InvF q;
  q.d = w_to_float(D, e);
  q.b = w_to_float(Bsq, e);
  q.qt2 = w_to_float(Qtsq, 2 * e);
  q.qb2 = w_to_float(norm(QdB * QdB), 3 * e);
  q.c = w_to_float(C, e);
  q.gf = (float)K.gf;
  {
    // (a root below 1e-6 D is left to the Wide steps)
    float w = w_to_float(Wp, e), last = 1.0f, hi = INFINITY;
    if (!(w > 1e-6f * q.d)) w = 1e-6f * q.d;
#pragma unroll 1
    for (int it = 0; it < INV_F32_MAXIT && last > 1e-5f; it++) {
      float f, df, n;
      if (inv_f32(q, w, f, df) < 0.99999f) {
        if (f > 0.0f) hi = w;
        n = w - f * inv_rcpf(df);
        if (!(n > 0.0f)) {
          if (it > 4) break;  // (no positive root, or one below FP32's noise)
          n = 0.5f * w;
        }
      } else {  // below the root
        n = (hi < INFINITY) ? 0.5f * (w + hi) : w + (w + q.d);
      }
      last = fabsf(n - w) * inv_rcpf(w);
      w = n;
    }
    const bool fine = last < 0.5f && w < 1e6f;
    if (fine)
      Wp = w_scale(wide_posf(w), -e);
    else if (Wp.s || Wp.m == 0)
      ok = false;
  }

  const Wide gf = wide_pos(K.gf);
  const Wide one = {1ull << 61, 0, -61};
  bool done = false;
  Wide iB, x, bsq, omv, rs, wmr;
#pragma unroll 1
  for (int it = 0; it < INV_WIDE_MAXIT && ok; it++) {
    const Wide W = norm(w_sum<1>(Wp, D));
    const Wide BW = norm(w_sum<1>(Bsq, W));
    const Wide ix = w_rcp(norm(BW * W));
    iB = norm(W * ix);              // 1/(B^2 + W)
    x = norm(QdB * norm(BW * ix));  // Q.B / W
    const Wide x2 = x * x;
    const Wide vsq = norm(norm(w_sum<1>(Qtsq, x2 * norm(w_sum<1>(Bsq, w_scale(W, 1))))) * norm(iB * iB));
    omv = norm(w_sum<1>(one, -vsq));
    ok = omv.s == 0 && omv.x >= -62 - 33;  // 1 - v^2 >= 2^-33
    if (!ok) break;
    rs = norm(w_rsqrt(omv));  // Lorentz factor
    const Wide sq = norm(omv * rs);
    // w - rho = W' (1 - v^2) - D v^2 sq / (1 + sq)
    wmr = w_sum<0>(Wp * omv, -(norm(norm(D * vsq) * sq) * w_rcp(norm(w_sum<1>(one, sq)))));
    bsq = w_sum<0>(Bsq * omv, x2);
    const Wide f = w_sum<2>(C, Wp, -(gf * norm(wmr)), -w_scale(bsq, -1));
    // (the sum shifts its largest term right by two bits)
    done = f.m < 1ull << w_min(w_max(f.x - 2, Bsq.x) - f.x + (62 - INV_RESIDUAL), 62);
    if (done) break;
    const float vf = w_to_float(omv, 0);
    const float df = inv_df(q, w_to_float(W, e), vf, inv_rsqrtf(vf), w_to_float(bsq, e));
    const Wide step = norm(f) * wide_posf(inv_rcpf(df));
    const Wide n = norm(w_sum<1>(Wp, -step));
    // below zero by no more than the derivative's error, the root is nearer to it than
    // that; by more there is none (u < 0)
    const bool above = n.s == 0 && n.m != 0;
    ok = df > 0.0f && (above || n.x < Wp.x - 12);
    Wp = above ? n : w_scale(Wp, -16);
  }
  ok = ok && done && (wmr.s == 0 || wmr.m == 0);
  if (!ok) return false;
  const Wide sq = norm(omv * rs), fac = norm(rs * iB);
  P[RHO] = w_to_double(D * sq);
  P[UU] = w_to_double(norm(wmr) * wide_pos(K.igam));
  P[U1] = w_to_double(fac * norm(w_sum<1>(Qt1, x * n1)));
  P[U2] = w_to_double(fac * norm(w_sum<1>(Qt2, x * n2)));
  P[U3] = w_to_double(fac * norm(w_sum<1>(Qt3, x * n3)));
#pragma unroll
  for (int i = 0; i < 3; i++) P[B1 + i] = b[i];
  bsq_out = w_to_double(bsq);
  lorentz_out = w_to_double(rs);
  return true;
#undef GCOV
#undef GDIA
#undef GCON
}

// U of a state P plus that of the drift-frame bounds' parcel (apply_floors_drift):
// density and internal energy dr, du, no field, the drift velocity utilde_d = f
// (utilde - q B) with q = (utilde.B)/B^2, f = 1/sqrt(1 + (utilde.B)^2/B^2), or the
// fluid's where B^2 <= bsq_min.  guess: W of a state with P's velocity and
// density and internal energy rho_f, u_f.
template <class GeoFn>
WIDE_FN void wide_drift_sum(const double P[NV], const GeoFn &geo, double gam, double dr, double du,
                            double bsq_min, double rho_f, double u_f, double U[NV], double &guess) {
  WideState s;
  wide_state<true>(P, geo, s);
  guess = w_fma(gam, u_f, rho_f) * w_to_double(s.g2);
  const double B2 = w_to_double(s.B2);
  Wide q = {0, 0, -2000}, f = {1ull << 62, 0, -62};
  const Wide one = {1ull << 61, 0, -61};
  if (B2 > bsq_min) {
    q = norm(s.bt * w_rcp(norm(s.B2)));
    f = norm(w_rsqrt(norm(w_sum<1>(one, s.bt * q))));
  }
  // the parcel's utilde, u_mu, u^t
  Wide vd[3], ud[4];
#pragma unroll
  for (int i = 0; i < 3; i++) {
    vd[i] = norm(f * norm(w_sum<1>(wide(P[U1 + i]), -(q * wide(P[B1 + i])))));
    ud[i + 1] = norm(f * norm(w_sum<1>(s.ucov[i + 1], -(q * s.Bcov[i + 1]))));
  }
  const Wide g2 = norm(w_sum<1>(one, ud[1] * vd[0], ud[2] * vd[1], ud[3] * vd[2]));
  const Wide gd = norm(g2 * w_rsqrt(g2));
  ud[0] = norm(w_sum<1>(wide(geo(G_GCOV + SY(0, 1))) * vd[0], wide(geo(G_GCOV + SY(0, 3))) * vd[2],
                        -(gd * wide_pos(geo(G_ALPHA)))));
  const Wide utd = norm(gd * wide_pos(geo(G_IALPHA)));
  // T^t_nu of both: (w u^t - k b^t) u_nu - k B_nu + w_d u^t_d u_d,nu, k = b^t / u^t
  const double gm1 = gam - 1.0;
  const Wide rho = wide(P[RHO]), pg = wide(gm1) * wide(P[UU]);
  const Wide w = norm(w_sum<2>(rho, wide(P[UU]), pg, s.bsq));
  const Wide k = norm(s.bt * s.iut);
  const Wide k1 = norm(w_sum<1>(w * s.ucon[0], -(k * s.bt))), nk = -k;
  const Wide kd = norm(wide(w_fma(gam, du, dr)) * utd);
  const Wide pt = w_sum<2>(pg, w_scale(s.bsq, -1), wide(gm1 * du));
  const Wide mass = w_sum<1>(rho * s.ucon[0], wide(dr) * utd), sg = wide_pos(geo(G_GDET));
  U[RHO] = w_to_double(norm(mass) * sg);
#pragma unroll
  for (int n = 0; n < 4; n++) {
    const Wide t = w_sum<1>(k1 * s.ucov[n], nk * s.Bcov[n], kd * ud[n]);
    U[UU + n] = w_to_double(norm(n ? t : w_sum<2>(t, pt, mass)) * sg);
  }
#pragma unroll
  for (int i = 0; i < 3; i++) U[B1 + i] = geo(G_GDET) * P[B1 + i];
}

}  // namespace grmhd
