// wide_face.cuh -- fluid state and LLF flux terms of one face state in Wide
// numbers (wide_num.cuh): the same formulas as fluid_state and prim_flux.
//
// BLK: the metric couples X2 to no other coordinate (g_{02} = g_{12} = g_{23} =
// g^{02} = g^{12} = g^{23} = 0, as in Minkowski and Kerr-Schild coordinates), so
// that the products with those components, zeros, are left out.
#pragma once

#include "grmhd_dev.cuh"
#include "wide_num.cuh"

namespace grmhd {

// What the LLF flux needs of a state.  In terms of the magnetic field's lowered
// components B_mu = g_{mu j} B^j,
//   b_mu = (B_mu + b^t u_mu) / u^t,  b^2 = (B_i B^i + (b^t)^2) / (u^t)^2,
// and the induction flux b^i u^d - b^d u^i = (B^i u^d - B^d u^i) / u^t, so that
// neither b^i nor b_mu need be formed.
struct WideState {
  Wide ucon[4], ucov[4];  // u^mu, u_mu
  Wide Bcov[4];           // B_mu
  Wide bt, bsq, iut;      // b^t, b^2, 1/u^t
  Wide g2, B2;            // Lorentz factor squared, B_i B^i
};

// geo(c): component c of the location's geometry (G_*), as a double
template <bool BLK, class GeoFn>
WIDE_FN void wide_state(const double P[NV], const GeoFn &geo, WideState &s) {
#define GCOV(m, n) wide(geo(G_GCOV + SY(m, n)))
#define GDIA(m) wide_pos(geo(G_GCOV + SY(m, m)))
#define GCON(m, n) wide(geo(G_GCON + SY(m, n)))
  const Wide v1 = wide(P[U1]), v2 = wide(P[U2]), v3 = wide(P[U3]);
  const Wide b1 = wide(P[B1]), b2 = wide(P[B2]), b3 = wide(P[B3]);
  {
    const Wide g11 = GDIA(1), g13 = GCOV(1, 3), g33 = GDIA(3), g22 = GDIA(2);
    if (BLK) {
      s.ucov[1] = w_sum<0>(g11 * v1, g13 * v3);
      s.ucov[2] = g22 * v2;
      s.ucov[3] = w_sum<0>(g13 * v1, g33 * v3);
      s.Bcov[1] = w_sum<0>(g11 * b1, g13 * b3);
      s.Bcov[2] = g22 * b2;
      s.Bcov[3] = w_sum<0>(g13 * b1, g33 * b3);
    } else {
      const Wide g12 = GCOV(1, 2), g23 = GCOV(2, 3);
      s.ucov[1] = w_sum<1>(g11 * v1, g12 * v2, g13 * v3);
      s.ucov[2] = w_sum<1>(g12 * v1, g22 * v2, g23 * v3);
      s.ucov[3] = w_sum<1>(g13 * v1, g23 * v2, g33 * v3);
      s.Bcov[1] = w_sum<1>(g11 * b1, g12 * b2, g13 * b3);
      s.Bcov[2] = w_sum<1>(g12 * b1, g22 * b2, g23 * b3);
      s.Bcov[3] = w_sum<1>(g13 * b1, g23 * b2, g33 * b3);
    }
  }
  const Wide one = {1ull << 61, 0, -61};
  const Wide g2 = norm(w_sum<1>(one, s.ucov[1] * v1, s.ucov[2] * v2, s.ucov[3] * v3));
  s.g2 = g2;
  const Wide rg = w_rsqrt(g2);
  const Wide gam = norm(g2 * rg);
  const Wide al = wide_pos(geo(G_ALPHA));
  const Wide ga = norm(gam * al);
  s.iut = norm(al * rg);
  s.bt = norm(w_sum<1>(b1 * s.ucov[1], b2 * s.ucov[2], b3 * s.ucov[3]));
  s.B2 = w_sum<1>(b1 * s.Bcov[1], b2 * s.Bcov[2], b3 * s.Bcov[3]);
  s.bsq = norm(norm(w_sum<1>(s.B2, s.bt * s.bt)) * (s.iut * s.iut));
  s.ucon[0] = gam * wide_pos(geo(G_IALPHA));
  s.ucon[1] = w_sum<1>(v1, -(ga * GCON(0, 1)));
  s.ucon[2] = BLK ? v2 : w_sum<1>(v2, -(ga * GCON(0, 2)));
  s.ucon[3] = w_sum<1>(v3, -(ga * GCON(0, 3)));
  if (BLK) {
    const Wide g01 = GCOV(0, 1), g03 = GCOV(0, 3);
    s.ucov[0] = w_sum<1>(g01 * v1, g03 * v3, -ga);
    s.Bcov[0] = w_sum<0>(g01 * b1, g03 * b3);
  } else {
    const Wide g01 = GCOV(0, 1), g02 = GCOV(0, 2), g03 = GCOV(0, 3);
    s.ucov[0] = w_sum<2>(g01 * v1, g02 * v2, g03 * v3, -ga);
    s.Bcov[0] = w_sum<1>(g01 * b1, g02 * b2, g03 * b3);
  }
#undef GCOV
#undef GDIA
#undef GCON
}

// f (F^dir + coef U) without sqrt(-g) of one state, rounded to double.  ee = rho +
// u + p + b^2, gm1 = gamma - 1; a state or coef that is not finite gives NaN.
// With uc = u^d + coef u^t, bc = b^d + coef b^t, k2 = bc / u^t:
//   T^d_nu + coef T^t_nu = (w uc - k2 b^t) u_nu - k2 B_nu (+ pressure),
//   B^i's row = (B^i uc - B^d u^i) / u^t, which is coef B^d for i = d.
WIDE_FN void wide_flux(const double P[NV], const WideState &s, double ee, double gm1, int dir,
                       double coef, double f, double out[NV]) {
  const Wide c = wide(coef), hg = wide(f);
  const Wide pt = w_sum<1>(wide(gm1) * wide(P[UU]), w_scale(s.bsq, -1));
  const Wide bd = wide(P[B1 - 1 + dir]);
  const Wide uc = norm(w_sum<1>(s.ucon[dir], c * s.ucon[0]));
  const Wide bcon = norm(w_sum<1>(bd, s.bt * s.ucon[dir])) * s.iut;
  const Wide k2 = norm(norm(w_sum<1>(bcon, c * s.bt)) * s.iut);
  const Wide k1 = norm(w_sum<1>(wide(ee) * uc, -(k2 * s.bt)));
  const Wide k3 = norm(uc * s.iut), k4 = -norm(bd * s.iut), nk2 = -k2;
  const Wide mf = wide(P[RHO]) * uc;
  Wide r[NV];
  r[RHO] = mf;
  r[UU] = w_sum<1>(k1 * s.ucov[0], nk2 * s.Bcov[0], c * pt, mf);
#pragma unroll
  for (int i = 1; i < 4; i++) {
    r[UU + i] = (i == dir) ? w_sum<1>(k1 * s.ucov[i], nk2 * s.Bcov[i], pt)
                           : w_sum<0>(k1 * s.ucov[i], nk2 * s.Bcov[i]);
    r[B1 - 1 + i] =
        (i == dir) ? c * bd : w_sum<0>(k3 * wide(P[B1 - 1 + i]), k4 * s.ucon[i]);
  }
  bool bad = !w_finite(coef) || !w_finite(P[RHO]);
  bad = bad || !w_finite(P[U1]) || !w_finite(P[U2]) || !w_finite(P[U3]);
  const bool bad1 = bad || !w_finite(P[UU]) || !w_finite(P[B1]) || !w_finite(P[B2]) || !w_finite(P[B3]);
  const double nan = w_double(0x7ffull << 52 | 1ull << 51);
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const double q = w_to_double(r[v] * hg);
    out[v] = ((v == RHO) ? bad : bad1) ? nan : q;
  }
}

}  // namespace grmhd
