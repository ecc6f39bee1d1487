// elec_bodies.cuh -- the electron entropies of a grid (paper, "Implementation
// Notes": the optional partition of dissipation between ions and electrons
// of Ressler et al. 2015 with five heating models, and the bound P_gas /
// rho^gamma < 3 of the bounds list when electron temperatures are evolved).
//
// kappa_tot = P_gas/rho^gamma and kappa_e = P_e/rho^gamma_e ride with the
// mass.  Per stage, after the fluid's kernels:
//   elec_recon_body<d> reconstructs both entropies at the two faces of every
//                      zone along d (as recon_body does the primitives);
//   elec_flux_body<d>  (after the face fluxes of every direction) forms their
//                      local Lax-Friedrichs flux from the weights that the
//                      face kernels (FP64, FP32 or float-float) stored;
//   fix_flux_body      zeroes them where the mass flux is zeroed (FP64 grids: the
//                      face kernels zero their weights there);
//   elec_post_body     (after the update, whose bounds wait for it) carries
//                      the entropies to the new state, heats the electrons by
//                      the model's share of the dissipation, applies the
//                      fluid's bounds (either frame), the entropy bound, the
//                      kappa_tot reset and the T_p/T_e bounds;
//   elec_fix_body      (after the fixup) gives a fixed-up zone the neighbour
//                      mean of kappa_e and the same closing steps.
#pragma once

#include "step_bodies.cuh"
#include "wide_pow.cuh"

namespace grmhd {

constexpr double KTOT_MAX = 3.0;          // P_gas / rho^gamma < 3
constexpr double ELEC_CLAMP = 1.0e20;     // T_p/T_e and beta_p within [1/C, C]
constexpr double MP_OVER_ME = 1836.15267343;
constexpr int FF_KTOT = 256;              // bound flag: u lowered for kappa_tot <= 3

// Powers of the density come from one logarithm per density value,
// rho^a = exp(a ln rho) (relative error about |a ln rho| x 1e-16, far below
// the step's rounding), instead of one pow() each.

// Heating share f_e of a zone (rho, u, kappa_e, b^2; lr = ln rho); models as
// documented with GRMHD_ELEC_* in grmhd.h.
static __device__ __noinline__ double elec_fraction(const StepArgs &A, double rho, double lr,
                                                    double u, double kel, double bsq) {
  if (A.elec == GRMHD_ELEC_CONSTANT) return A.fel_const;
  const double ue = kel * exp(A.game * lr) / (A.game - 1.0);
  const double Te = fabs((A.game - 1.0) * ue / rho);
  const double Tp = fabs((A.gamp - 1.0) * (u - ue) / rho);
  double trat = (Te > 0.0) ? Tp / Te : ELEC_CLAMP;  // T_p / T_e
  trat = fmin(fmax(trat, 1.0 / ELEC_CLAMP), ELEC_CLAMP);
  double beta = (bsq > 0.0) ? 2.0 * rho * Tp / bsq : ELEC_CLAMP;
  beta = fmin(fmax(beta, 1.0 / ELEC_CLAMP), ELEC_CLAMP);
  switch (A.elec) {
    case GRMHD_ELEC_KAWAZURA: {
      const double qiqe = 35.0 / (1.0 + pow(beta / 15.0, -1.4) * exp(-0.1 / trat));
      return 1.0 / (1.0 + qiqe);
    }
    case GRMHD_ELEC_WERNER: {
      const double s = bsq / rho;
      return 0.25 * (1.0 + sqrt((s / 5.0) / (2.0 + s / 5.0)));
    }
    case GRMHD_ELEC_ROWAN: {
      const double sw = bsq / (rho + A.gam * u);
      const double r = fmin(4.0 * sw * beta, 1.0);  // beta_p / beta_max
      return 0.5 * exp(-pow(1.0 - r, 3.3) / (1.0 + 1.2 * pow(sw, 0.7)));
    }
    case GRMHD_ELEC_SHARMA: {
      const double qeqi = 0.33 * sqrt(1.0 / trat);
      return qeqi / (1.0 + qeqi);
    }
    case GRMHD_ELEC_HOWES: {
      const double lt = log10(trat);
      const double c2 = (trat > 1.0) ? 1.6 / trat : 1.2 / trat;
      const double c3 = (trat > 1.0) ? 18.0 + 5.0 * lt : 18.0;
      const double bx = pow(beta, 2.0 - 0.2 * lt);
      const double qiqe = 0.92 * (c2 * c2 + bx) / (c3 * c3 + bx) * sqrt(MP_OVER_ME * trat) *
                          exp(-1.0 / beta);
      return 1.0 / (1.0 + qiqe);
    }
  }
  return 0.0;
}

// kappa_e after the heating (elec_post_body) of a zone in FP64
static __device__ __noinline__ double elec_heat(const StepArgs &A, double rho_s, double u_s,
                                                double kel_s, double bsq_s, double rho_n,
                                                double u_n, const double kn[2]) {
  const double ls = log(rho_s);
  const double fel = elec_fraction(A, rho_s, ls, u_s, kel_s, bsq_s);
  const double ktot = (A.gam - 1.0) * u_n / exp(A.gam * log(rho_n));
  return kn[1] + fel * (A.game - 1.0) / (A.gam - 1.0) * exp((A.gam - A.game) * ls) *
                     (ktot - kn[0]);
}

// The closing steps of a zone once the fluid's bounds are done: u lowered
// to P_gas/rho^gamma = 3 where it exceeds that (with the bounds on),
// kappa_tot reset to (gamma - 1) u / rho^gamma, kappa_e held to
// tpte_min <= T_p/T_e <= tpte_max, i.e. within kappa_tot rho^(gamma -
// gamma_e) / ((gamma - 1)/(gamma_e - 1) + R (gamma - 1)/(gamma_p - 1)) at
// R = tpte_max .. tpte_min (a kappa_e that is not a number takes the lower).
// lr = ln P[RHO].
static __device__ __noinline__ int elec_close(const StepArgs &A, double P[NV], double K[2],
                                              double lr) {
  int fl = 0;
  const double g1 = A.gam - 1.0;
  const double rg = exp(A.gam * lr);
  if (A.floors_on) {
    const double kt = g1 * P[UU] / rg;
    if (kt > KTOT_MAX) {
      P[UU] = KTOT_MAX * rg / g1;
      fl = FF_KTOT;
    }
  }
  K[0] = g1 * P[UU] / rg;
  const double a = g1 / (A.game - 1.0), b = g1 / (A.gamp - 1.0);
  const double kk = K[0] * exp((A.gam - A.game) * lr);
  const double kmax = kk / (a + A.tpte_min * b);
  const double kmin = kk / (a + A.tpte_max * b);
  double kel = K[1];
  if (!(kel == kel)) kel = kmin;
  K[1] = fmin(fmax(kel, kmin), kmax);
  return fl;
}

// ---------------------------------------------------------------------------
// The same in Wide numbers (wide_num.cuh, wide_pow.cuh).  With log, exp, pow and
// the divisions in FP64 the pass after the update was bound by that unit's 460
// instructions a zone: 0.84 ms per launch on a 96^3 grid with Kawazura's model, 0.13
// now.  Zones whose state leaves the range the powers are taken in (densities within
// 2^+-52, energies and entropies within 2^+-100) take the FP64 form above; b^2 may be
// anything finite, since beta is held within 1e+-20 (rounding leaves b^2 of 1e-40 and
// less around a magnetised region).
// ---------------------------------------------------------------------------
constexpr int ELEC_RHO_RANGE = 52, ELEC_RANGE = 100;

// elec_fraction's heating of kn[1]: the advected entropies kn, the source state s,
// the new state n; ln: log2 rho_n, kt: kappa_tot of the new state.  False: take the
// FP64 form.
__device__ __forceinline__ bool elec_heat_wide(const StepArgs &A, double rho_s, double u_s,
                                               double kel_s, double bsq_s, double rho_n,
                                               double u_n, Wide kn[2], s64 &ln, Wide &kt) {
  if (!w_within(rho_s, ELEC_RHO_RANGE) || !w_within(rho_n, ELEC_RHO_RANGE) ||
      !w_within(u_s, ELEC_RANGE) || !w_within(u_n, ELEC_RANGE) || !w_within(kel_s, ELEC_RANGE) ||
      !w_finite(bsq_s))
    return false;
  const s64 l = w_log2(wide_pos(rho_s));
  const Wide ls = w_log_num(l);
  Wide fel;
  if (A.elec == GRMHD_ELEC_KAWAZURA) {
    fel = wide_kawazura(A.game, A.gamp, A.ek.ige, rho_s, ls, u_s, kel_s, bsq_s);
  } else {
    const double f = elec_fraction(A, rho_s, (double)l * (0.6931471805599453 * 0x1p-55), u_s,
                                   kel_s, bsq_s);
    if (!w_finite(f)) return false;
    fel = wide(f);
  }
  ln = w_log2(wide_pos(rho_n));
  kt = wide_pos(A.gm1) * wide_pos(u_n) * w_exp2(-(w_log_num(ln) * wide_pos(A.gam)));
  const Wide heat = fel * wide_pos(A.ek.c) * w_exp2(ls * wide(A.ek.dgam)) *
                    norm(w_sum<0>(kt, -kn[0]));
  kn[1] = w_sum<0>(kn[1], heat);
  return true;
}

// elec_close from Wide entropies: moved: the bounds changed P (rho0: its density
// before), else ln and kt hold.  False: take the FP64 form (P unchanged).
__device__ __forceinline__ bool elec_close_wide(const StepArgs &A, double P[NV], bool moved,
                                                double rho0, s64 ln, Wide kt, const Wide &kel,
                                                double K[2], int &fl) {
  if (!w_within(P[RHO], ELEC_RHO_RANGE) || !w_within(P[UU], ELEC_RANGE)) return false;
  fl = 0;
  if (moved && P[RHO] != rho0) ln = w_log2(wide_pos(P[RHO]));
  const Wide l = w_log_num(ln);
  const Wide rg = w_exp2(-(l * wide_pos(A.gam)));
  if (moved) kt = wide_pos(A.gm1) * wide_pos(P[UU]) * rg;
  K[0] = w_to_double(kt);
  if (A.floors_on && less(KTOT_MAX, K[0])) {
    P[UU] = w_to_double(wide_pos(KTOT_MAX) * wide_pos(A.ek.ig) * w_rcp(norm(rg)));
    fl = FF_KTOT;
    kt = wide_pos(A.gm1) * wide(P[UU]) * rg;
    K[0] = w_to_double(kt);
  }
  const Wide kk = norm(kt * w_exp2(l * wide(A.ek.dgam)));
  const Wide dmin = wide_pos(A.ek.dmin), dmax = wide_pos(A.ek.dmax), k = norm(kel);
  if (w_sum<1>(k * dmin, -kk).s)
    K[1] = w_to_double(kk * w_rcp(dmin));
  else if (w_sum<1>(kk, -(k * dmax)).s)
    K[1] = w_to_double(kk * w_rcp(dmax));
  else
    K[1] = w_to_double(k);
  return true;
}

// Zone-centric reconstruction of both entropies along DIR (the zones of
// recon_body): KLf = value at the zone's low face, KRf = at its high face,
// [2][ntot] each.
template <int DIR>
__device__ __forceinline__ void elec_recon_body(const StepArgs &A, const double *__restrict__ K,
                                                double *__restrict__ KLf,
                                                double *__restrict__ KRf, long long t) {
  const Dims &D = A.D;
  const int e0 = D.n[0] + 2, e1 = D.n[1] + 2;
  if (t >= n_recon(D, A.flat3)) return;
  const Idx3 q3 = unflatten(t, e0, e1);
  const int i = NG - 1 + q3.i, j = NG - 1 + q3.j, k = (A.flat3 ? NG : NG - 1) + q3.k;
  const long long c = zid(D, i, j, k);
  const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const double *p = K + q * D.ntot + c;
    double lo, hi;
    if (A.recon == 1) {
      weno5_wide_pair(__ldg(p - 2 * st), __ldg(p - st), __ldg(p), __ldg(p + st), __ldg(p + 2 * st),
                      lo, hi);
    } else {
      const double x1 = __ldg(p), h = mc_half_slope(x1 - __ldg(p - st), __ldg(p + st) - x1);
      lo = x1 - h;
      hi = x1 + h;
    }
    KLf[q * D.ntot + c] = lo;
    KRf[q * D.ntot + c] = hi;
  }
}

// Entropy fluxes of one face along DIR (the face box of face_body):
// F_K = w_L K_L + w_R K_R with K_L the high-face value of zone c-1, K_R the
// low-face value of zone c, and the weights the face kernel of the grid's
// precision stored, w_L = sqrt(-g)/2 rho_L (u^d_L + c u^t_L),
// w_R = sqrt(-g)/2 rho_R (u^d_R - c u^t_R) (c: the face's LLF speed), so
// that F_K is the LLF combination of rho u^d K and rho u^t K.
template <int DIR>
__device__ __forceinline__ void elec_flux_body(const StepArgs &A, const double *__restrict__ KLf,
                                               const double *__restrict__ KRf,
                                               double *__restrict__ FK, long long t) {
  const Dims &D = A.D;
  int lo[3], ext[3];
  face_box(D, DIR, A.flat3, lo, ext);
  if (t >= (long long)ext[0] * ext[1] * ext[2]) return;
  const Idx3 q3 = unflatten(t, ext[0], ext[1]);
  const int i = lo[0] + q3.i, j = lo[1] + q3.j, k = lo[2] + q3.k;
  const long long c = zid(D, i, j, k), N = D.ntot;
  const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
  const double wl = A.elec_w[(2 * DIR) * N + c], wr = A.elec_w[(2 * DIR + 1) * N + c];
#pragma unroll
  for (int q = 0; q < 2; q++) FK[q * N + c] = wl * KRf[q * N + c - st] + wr * KLf[q * N + c];
}

// After the update: the entropies carried to the new state, U_K = U_rho(P_i)
// K_i - dt' div F_K and kappa_adv = U_K / U_rho(new), U_rho(new) = U_rho(P_i)
// - dt' div F_rho; then, in a zone whose inversion succeeded (Pout holds its
// unbounded state), the heating kappa_e = kappa_e,adv + f_e (gamma_e - 1) /
// (gamma - 1) rho_s^(gamma - gamma_e) ((gamma - 1) u/rho^gamma -
// kappa_tot,adv) with f_e from the source state P_s, the fluid's bounds and
// the closing steps.  U_rho(P_i) is what the update keeps of U(P^n); scratch holds
// b^2 of P_s, and b^2 and the Lorentz factor of the unbounded state.  Every thread
// of the block must call it (warp counters).
__device__ __forceinline__ void elec_post_body(const StepArgs &A, const double *Ps, double *Pout,
                                               const double *__restrict__ F1,
                                               const double *__restrict__ F2,
                                               const double *__restrict__ F3,
                                               const double *__restrict__ FK1,
                                               const double *__restrict__ FK2,
                                               const double *__restrict__ FK3, const double *Ki,
                                               const double *Ks, double *Kout,
                                               const double *__restrict__ Ucache,
                                               const double *__restrict__ scratch,
                                               const int *__restrict__ pflag, int *fflag,
                                               double dtfac, long long t) {
  const Dims &D = A.D;
  const double dt = A.clk->dt;
  if (!less(0.0, dt)) return;
  const double dtp = dtfac * dt;
  const bool in = t < n_update(D);
  const Column q3 = column_of(in ? t : t & 31, (int)(t & 31), 32, D.n[0], D.n[1], D.n[2]);
  const bool active = in && q3.active;
  int ff = 0;
  if (active) {
    const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
    const long long c = zid(D, i, j, k), N = D.ntot;
    const long long ij = (long long)j * D.s[0] + i;
    const double rho_s = Ps[RHO * N + c], u_s = Ps[UU * N + c], Uri = Ucache[RHO * N + c];
    const double Urn = fma(-dtp, flux_div(A, F1, F2, F3, RHO * N + c), Uri);
    double num[2], kn[2];
#pragma unroll
    for (int q = 0; q < 2; q++) {
      const long long oq = q * N + c;
      num[q] = fma(-dtp, flux_div(A, FK1, FK2, FK3, oq), Uri * Ki[oq]);
    }
    const bool in_range = A.ek.wide && w_within(Urn, ELEC_RANGE) &&
                          w_within(fabs(num[0]), 2 * ELEC_RANGE) &&
                          w_within(fabs(num[1]), 2 * ELEC_RANGE);
    Wide kw[2];
    if (in_range) {
      const Wide r = w_rcp(wide_pos(Urn));
#pragma unroll
      for (int q = 0; q < 2; q++) {
        kw[q] = wide(num[q]) * r;
        kn[q] = w_to_double(kw[q]);
      }
    } else {
      kn[0] = num[0] / Urn;
      kn[1] = num[1] / Urn;
    }
    if (pflag[c] == 0) {
      double pn[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) pn[v] = Pout[v * N + c];
      const double rho_n = pn[RHO], u_n = pn[UU], kel_s = Ks[N + c];
      const double bsq_s = scratch[SCR_BSQ_S * N + c];
      s64 ln = 0;
      Wide kt;
      const bool wide_zone =
          in_range && elec_heat_wide(A, rho_s, u_s, kel_s, bsq_s, rho_n, u_n, kw, ln, kt);
      if (!wide_zone) kn[1] = elec_heat(A, rho_s, u_s, kel_s, bsq_s, rho_n, u_n, kn);
      if (A.floors_on) {
        const double bsq = scratch[SCR_BSQ * N + c], lor = scratch[SCR_LORENTZ * N + c];
        ff = A.floor_drift ? floors_drift(A, ij, pn, bsq, lor) : floors_fluid(A, ij, pn, bsq, lor);
      }
      int fk;
      if (!wide_zone || !elec_close_wide(A, pn, ff != 0, rho_n, ln, kt, kw[1], kn, fk)) {
        if (wide_zone) kn[1] = w_to_double(kw[1]);
        double p[NV];
        p[RHO] = pn[RHO];
        p[UU] = pn[UU];
        fk = elec_close(A, p, kn, log(p[RHO]));
        pn[UU] = p[UU];
      }
      ff |= fk;
#pragma unroll
      for (int v = 0; v < NV; v++) Pout[v * N + c] = pn[v];
      fflag[c] = ff;
    }
    Kout[c] = kn[0];
    Kout[N + c] = kn[1];
  }
  count_warp(active && ff != 0, &A.clk->counters[1]);
}

// After the fixup: a fixed-up zone takes the mean kappa_e of the same
// neighbours and the closing steps (its bound flags gain FF_KTOT where u
// was lowered).  Every thread of the block must call it (warp counters).
__device__ __forceinline__ void elec_fix_body(const StepArgs &A, double *P, double *K,
                                              const int *__restrict__ pflag, int *fflag,
                                              long long t) {
  const Dims &D = A.D;
  if (!less(0.0, A.clk->dt)) return;
  for_failed_zones(A, pflag, t, [&](int i, int j, int k) {
    const long long c = zid(D, i, j, k), N = D.ntot;
    double sum = 0.0;
    int cnt = 0;
    for (int dk = -1; dk <= 1; dk++)
      for (int dj = -1; dj <= 1; dj++)
        for (int di = -1; di <= 1; di++) {
          if (di == 0 && dj == 0 && dk == 0) continue;
          const int ii = i + di, jj = j + dj, kk = k + dk;
          if (ii < NG - A.xlo[0] || ii >= D.n[0] + NG + A.xhi[0] || jj < NG - A.xlo[1] ||
              jj >= D.n[1] + NG + A.xhi[1] || kk < NG - A.xlo[2] || kk >= D.n[2] + NG + A.xhi[2])
            continue;
          const long long nb = zid(D, ii, jj, kk);
          if (pflag[nb] != 0) continue;
          sum += K[N + nb];
          cnt++;
        }
    if (cnt == 0) return 0;
    double p[NV], kn[2] = {0.0, sum / (double)cnt};
#pragma unroll
    for (int v = 0; v < NV; v++) p[v] = P[v * N + c];
    const int f = elec_close(A, p, kn, log(p[RHO]));
    P[UU * N + c] = p[UU];
    K[c] = kn[0];
    K[N + c] = kn[1];
    const int hit = f && fflag[c] == 0;
    if (f) fflag[c] |= f;
    return hit;
  });
}

}  // namespace grmhd
