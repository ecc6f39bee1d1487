"""The 1D_W inversion in Wide numbers (csrc/wide_update.cuh), built for the host,
at Lorentz factors up to 50 and beyond, against the root of the same conserved vector
in 40 decimal digits.

Tolerances.  Every quantity that the 1D_W function f(W') sums is a product chain rounded
to 2^-53 (the conserved vector's own rounding does not count: the root is that of the
rounded one), a dozen roundings of terms no larger than W + B^2, so that W is off by
16 x 2^-53 (W + B^2) / f'.  rho = D sqrt(1 - v^2) and u follow with d(1 - v^2) = 2 (v^2 W
+ (Q.B/W)^2) / (B^2 + W) dW/W plus 16 x 2^-53 of v^2 itself; FP64 numbers leave as much."""
import ctypes
import decimal
import subprocess

import numpy as np
import pytest

import oracle
from paper_2110_10191_gb300 import build as _build

U53 = 2.0 ** -53
SRC = r"""
#include "wide_update.cuh"
using namespace grmhd;
extern "C" int invert(const double *U, const double *g, double gam, double guess, int blk,
                      double *P, double *bl) {
  GasK K;
  K.gam = gam; K.igam = 1.0 / gam; K.gf = (gam - 1.0) / gam;
  auto geo = [&](int k) { return g[k]; };
  return blk ? wide_invert<true>(U, geo, K, guess, P, bl[0], bl[1])
             : wide_invert<false>(U, geo, K, guess, P, bl[0], bl[1]);
}
"""
SY = [(m, n) for m in range(4) for n in range(m, 4)]
IDX = {}
for _q, (_m, _n) in enumerate(SY):
    IDX[_m, _n] = IDX[_n, _m] = _q


@pytest.fixture(scope="module")
def wide(tmp_path_factory):
    d = tmp_path_factory.mktemp("invert")
    (d / "w.cu").write_text(SRC)
    so = str(d / "w.so")
    subprocess.run([_build.nvcc(), "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", _build.CSRC, "-o", so, str(d / "w.cu")], check=True)
    lib = ctypes.CDLL(so)

    def call(U, g, gam, guess, blk=1):
        P, bl = np.zeros(8), np.zeros(2)
        p = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
        U, g = np.ascontiguousarray(U), np.ascontiguousarray(g)
        ok = lib.invert(p(U), p(g), ctypes.c_double(gam), ctypes.c_double(guess), blk, p(P), p(bl))
        return ok, P, bl
    return call


def _point(kind, rng):
    X = (0.0, float(np.log(10.0 ** rng.uniform(0.2, 1.69))), float(rng.uniform(0.02, 0.98)), 0.0)
    q = oracle.geom_at(kind, 0.9375, 0.3, X)
    gi, al = q["gcon"], q["alpha"]
    return X, q["gcov"], np.array([q["gcov"][m, n] for m, n in SY] + [gi[m, n] for m, n in SY] +
                                  [q["gdet"], al, 1 / al, 1 / q["gdet"], (1 + 1 / gi[0, 0]) / (1 + al)])


def _state(gcov, rng, X, kind, lorentz, uor, sigma, along):
    """density 1e-6 .. 1, u = uor rho, b^2 = sigma rho; the field along the flow but for
    a share `along` of a random direction (None: random)."""
    h = gcov[1:, 1:]
    d = rng.normal(size=3)
    d /= np.sqrt(d @ h @ d)
    P = np.zeros(8)
    P[0] = 10.0 ** rng.uniform(-6, 0)
    P[1] = P[0] * uor
    P[2:5] = np.sqrt(lorentz ** 2 - 1) * d
    if sigma:
        b = rng.normal(size=3)
        b /= np.sqrt(b @ h @ b)
        P[5:8] = b if along is None else d + along * b
        bsq = oracle.state_at(kind, 0.9375, 0.3, X, P)["bsq"]
        P[5:8] *= np.sqrt(sigma * P[0] / bsq)
    return P


class Root:
    """rho, u of the conserved vector U in 40 digits, from a W' near the root, and the
    tolerances of both."""

    def __init__(self, U, g, gam, wp):
        with decimal.localcontext() as ctx:
            ctx.prec = 40
            D = decimal.Decimal
            G = [D(float(x)) for x in g]
            u = [D(float(x)) for x in U]
            al, igd = G[21], G[23]
            gi = lambda m, n: G[10 + IDX[m, n]]  # noqa: E731
            n = [al * D(float(U[5 + i]) * float(g[23])) for i in range(3)]
            Q = [al * igd * u[2 + i] for i in range(3)]
            rho_d = u[0] * al * igd
            cQ = sum(gi(0, i + 1) * Q[i] for i in range(3))
            qpn = (u[1] - G[24] * u[0]) * igd - al * cQ
            Qt = [sum(gi(i + 1, j + 1) * Q[j] for j in range(3)) + gi(0, i + 1) * al * al * cQ
                  for i in range(3)]
            Q2 = sum(Qt[i] * Q[i] for i in range(3))
            QB = sum(Q[i] * n[i] for i in range(3))
            B2 = sum(G[IDX[i + 1, j + 1]] * n[i] * n[j] for i in range(3) for j in range(3))
            gf = D((gam - 1.0) / gam)
            wp = D(float(wp))
            for it in range(60):
                W = wp + rho_d
                x2 = (QB / W) ** 2
                BW = B2 + W
                vsq = (Q2 + x2 * (B2 + 2 * W)) / (BW * BW)
                omv = 1 - vsq
                if omv <= 0:
                    wp += W
                    continue
                sq = omv.sqrt()
                wmr = wp * omv - rho_d * vsq * sq / (1 + sq)
                f = qpn + wp - gf * wmr + (1 + vsq) * B2 / 2 - x2 / 2
                q = (vsq * W + x2) / BW  # -W/2 dv^2/dW
                df = 1 - gf * (omv + 2 * q - q * rho_d / (sq * W)) + (x2 - B2 * q) / W
                wp -= f / df
                if abs(f / df) < abs(wp) * D("1e-32"):
                    break
            assert it < 59
            dw = 16 * U53 * float((W + B2) / abs(df)) / float(W)  # relative error of W
            domv = 2 * float(q) * dw + 16 * U53
            self.rho = float(rho_d * sq)
            self.u = float(wmr / D(gam))
            self.lorentz = float(1 / sq)
            self.tol_rho = domv / float(omv) / 2
            # u = ((W' + D)(1 - v^2) - D sq) / gamma
            self.tol_u = (float(W) * (domv + dw * float(omv)) + float(rho_d) * float(sq) * self.tol_rho) / \
                gam / max(self.u, 1e-300)


def _check(wide, rng, gam, lorentz, uor, sigma, along, off, count, kind):
    """worst (rho, u) errors in units of their tolerances, share of states answered"""
    worst, answered = np.zeros(2), 0
    for _ in range(count):
        X, gcov, g = _point(kind, rng)
        lf = lorentz[0] * (lorentz[1] / lorentz[0]) ** rng.uniform()
        P = _state(gcov, rng, X, kind, lf, 10.0 ** rng.uniform(*uor),
                   10.0 ** rng.uniform(*sigma) if sigma else 0.0, along)
        U = oracle.prim_to_flux(kind, 0.9375, 0.3, X, gam, P, 0)
        W = (P[0] + gam * P[1]) * lf * lf
        ok, out, bl = wide(U, g, gam, W * np.exp(rng.uniform(-off, off)))
        if not ok:
            continue
        answered += 1
        r = Root(U, g, gam, W - U[0] * g[21] * g[23])
        worst = np.maximum(worst, [abs(out[0] / r.rho - 1) / r.tol_rho, abs(out[1] / r.u - 1) / r.tol_u])
    return worst, answered / count


@pytest.mark.parametrize("gam", [13.0 / 9.0, 5.0 / 3.0])
@pytest.mark.parametrize("kind", [0, 1])
def test_the_state_is_the_last_iterates(wide, gam, kind):
    """Unmagnetised, Lorentz factors where the iteration takes all its steps: what comes
    back belongs to the W' at which it stopped, not to the one before."""
    worst, _ = _check(wide, np.random.default_rng(11), gam, (8.0, 20.0), (-2, 0), None, None,
                      0.3, 1500, kind)
    assert worst.max() <= 1.0


@pytest.mark.parametrize("lorentz", [(1.0, 8.0), (20.0, 50.0), (50.0, 1000.0)])
@pytest.mark.parametrize("sigma,along", [(None, None), ((-4, 2.6), None), ((0, 4), 0.1)])
@pytest.mark.parametrize("gam", [4.0 / 3.0, 5.0 / 3.0])
def test_an_answer_is_the_root(wide, gam, sigma, along, lorentz):
    """Any Lorentz factor and magnetisation, a guess off by up to e: no answer, or
    the root's."""
    seed = int(lorentz[1]) + 7 * (sigma is None) + 3 * (along is None)
    worst, _ = _check(wide, np.random.default_rng(seed), gam, lorentz, (-6, 0.5), sigma, along, 1.0,
                      400, seed % 2)
    assert worst.max() <= 1.0


def test_no_answer_from_a_derivative_that_overflows(wide):
    """Lorentz factor 1000: 1 - v^2 rounds to zero in FP32."""
    g = np.array([-1.0, 0, 0, 0, 1, 0, 0, 1, 0, 1] * 2 + [1.0, 1.0, 1.0, 1.0, 0.0])
    P = np.array([1.0, 2.004076452014, 927.43315163681, 368.26909591672, -65.15076572658,
                  733.51245163870, -657.53838453502, 172.05451506445])
    X, gam = (0.0, 0.0, 0.0, 0.0), 4.0 / 3.0
    U = oracle.prim_to_flux(0, 0.0, 0.3, X, gam, P, 0)
    ok, out, bl = wide(U, g, gam, 3671075.19870)
    if ok:
        r = Root(U, g, gam, (P[0] + gam * P[1]) * (1 + P[2:5] @ P[2:5]) - U[0])
        assert abs(out[0] / r.rho - 1) <= r.tol_rho and abs(out[1] / r.u - 1) <= r.tol_u


@pytest.mark.parametrize("sigma", [None, (-4, 2.6)])
@pytest.mark.parametrize("gam", [4.0 / 3.0, 13.0 / 9.0, 5.0 / 3.0])
def test_no_further_off_than_fp64(wide, gam, sigma):
    """Over Lorentz factors up to the bound of 50, the worst errors of rho and u are no
    larger than those of the FP64 iteration on the same conserved vectors."""
    rng = np.random.default_rng(5)
    worst = np.zeros((2, 2))
    for _ in range(600):
        X, gcov, g = _point(0, rng)
        lf = 50.0 ** rng.uniform()
        P = _state(gcov, rng, X, 0, lf, 10.0 ** rng.uniform(-4, 0),
                   10.0 ** rng.uniform(*sigma) if sigma else 0.0, None)
        U = oracle.prim_to_flux(0, 0.9375, 0.3, X, gam, P, 0)
        off = np.exp(rng.uniform(-0.3, 0.3))
        W = (P[0] + gam * P[1]) * lf * lf
        ok, out, _ = wide(U, g, gam, W * off)
        rc, P64 = oracle.cons_to_prim(0, 0.9375, 0.3, X, gam, U, P * np.array([off] * 2 + [1] * 6))
        if not ok or rc:
            continue
        r = Root(U, g, gam, W - U[0] * g[21] * g[23])
        for q, p in enumerate((out, P64)):
            worst[q] = np.maximum(worst[q], [abs(p[0] / r.rho - 1), abs(p[1] / r.u - 1)])
    assert (worst[0] <= worst[1]).all(), worst


@pytest.mark.parametrize("lorentz", [(1.0, 8.0), (8.0, 20.0), (20.0, 50.0)])
@pytest.mark.parametrize("sigma", [None, (-4, 2.6)])
@pytest.mark.parametrize("gam", [4.0 / 3.0, 13.0 / 9.0, 5.0 / 3.0])
def test_relativistic_states_are_answered(wide, gam, sigma, lorentz):
    """From guesses off by up to e, at most 1% are left to the FP64 iteration."""
    rng = np.random.default_rng(17)
    count, answered = 500, 0
    for _ in range(count):
        X, gcov, g = _point(0, rng)
        lf = lorentz[0] * (lorentz[1] / lorentz[0]) ** rng.uniform()
        P = _state(gcov, rng, X, 0, lf, 10.0 ** rng.uniform(-6, 0),
                   10.0 ** rng.uniform(*sigma) if sigma else 0.0, None)
        U = oracle.prim_to_flux(0, 0.9375, 0.3, X, gam, P, 0)
        answered += wide(U, g, gam, (P[0] + gam * P[1]) * lf * lf * np.exp(rng.uniform(-1, 1)))[0]
    assert answered >= 0.99 * count
