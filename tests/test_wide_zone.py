"""U(P), the stress-energy tensor (by the geometric source it gives) and the 1D_W
inversion in Wide numbers
(csrc/wide_update.cuh), built for the host, against the oracle's FP64.

Tolerances.  U and S: sums of a dozen products, each rounded to 2^-53 on the
oracle's side, of metric components whose 4x4 inverse carries 2^-53 times the
metric's condition (g_11 and g_22 reach r^2 and (pi r)^2, r <= 50: 1e4 and more),
1e4 x 2^-53 = 1e-12 of the largest term.  The inversion is given the oracle's U,
rounded to 2^-53 of gamma^2 (rho + u + b^2), from which u is recovered: the
relative error of u is that ratio's, times 64 for the dozen operations on it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2110_10191_gb300 import build as _build

GAM = 4.0 / 3.0
U53 = 2.0 ** -53
SRC = r"""
#include "wide_update.cuh"
using namespace grmhd;
extern "C" void tensor(const double *P, const double *g, int blk, double *U, double (*T)[4],
                       double *g2) {
  auto geo = [&](int k) { return g[k]; };
  double b2;
  if (blk) wide_tensor<true, true>(P, geo, GAM - 1.0, U, T, *g2, b2);
  else wide_tensor<false, true>(P, geo, GAM - 1.0, U, T, *g2, b2);
}
extern "C" int invert(const double *U, const double *g, double guess, int blk, double *P,
                      double *bl) {
  GasK K;
  K.gam = GAM; K.igam = 1.0 / GAM; K.gf = (GAM - 1.0) / GAM;
  auto geo = [&](int k) { return g[k]; };
  return blk ? wide_invert<true>(U, geo, K, guess, P, bl[0], bl[1])
             : wide_invert<false>(U, geo, K, guess, P, bl[0], bl[1]);
}
"""


@pytest.fixture(scope="module")
def wide(tmp_path_factory):
    d = tmp_path_factory.mktemp("zone")
    (d / "w.cu").write_text("#define GAM (4.0 / 3.0)\n" + SRC)
    so = str(d / "w.so")
    subprocess.run([_build.nvcc(), "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", _build.CSRC, "-o", so, str(d / "w.cu")], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return ctypes.c_void_p(a.ctypes.data)


def _point(kind, rng):
    X = (0.0, float(np.log(10.0 ** rng.uniform(0.2, 1.69))), float(rng.uniform(0.02, 0.98)), 0.0)
    q = oracle.geom_at(kind, 0.9375, 0.3, X)
    sy = [(m, n) for m in range(4) for n in range(m, 4)]
    gi, al = q["gcon"], q["alpha"]
    g = np.array([q["gcov"][m, n] for m, n in sy] + [gi[m, n] for m, n in sy] +
                 [q["gdet"], al, 1 / al, 1 / q["gdet"], (1 + 1 / gi[0, 0]) / (1 + al)])
    return X, q["gcov"], g, q["conn"]


def _state(g, rng, it):
    lv = np.sqrt(np.diag(g)[1:])
    P = np.zeros(8)
    P[0] = 10.0 ** rng.uniform(-12, 0)
    P[1] = P[0] * 10.0 ** rng.uniform(-4, 2)
    if it % 11:
        P[2:5] = 10.0 ** rng.uniform(-8, 0.7) * rng.normal(size=3) / lv
    if it % 7:
        P[5:8] = np.sqrt(P[0]) * 10.0 ** rng.uniform(-4, 1.2) * rng.normal(size=3) / lv
    return P


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("blk", [0, 1])
def test_source_and_inversion(wide, kind, blk):
    rng = np.random.default_rng(3 + kind)
    for it in range(400):
        X, gcov, g, conn = _point(kind, rng)
        P = _state(gcov, rng, it)
        U, T, g2, out, bl = np.zeros(8), np.zeros((4, 4)), np.zeros(1), np.zeros(8), np.zeros(2)
        wide.tensor(_p(P), _p(g), blk, _p(U), _p(T), _p(g2))
        S = g[20] * np.einsum("kl,lnk->n", T, conn)
        Uo, So = oracle.prim_to_flux(kind, 0.9375, 0.3, X, GAM, P, 0), oracle.source_at(kind, 0.9375, 0.3, X, GAM, P)
        scale = np.abs(Uo[:5]).max()
        assert np.abs(U[:5] - Uo[:5]).max() <= 1e-12 * scale
        assert abs(U[0] - Uo[0]) <= 64 * U53 * abs(Uo[0])
        assert np.abs(S - So[1:5]).max() <= 1e-12 * max(np.abs(conn).max() * scale * np.abs(gcov).max(), 0.0)
        gam2 = g2[0]
        guess = (P[0] + GAM * P[1]) * gam2 * rng.uniform(0.9, 1.1)
        assert wide.invert(_p(Uo), _p(g), ctypes.c_double(guess), blk, _p(out), _p(bl)) == 1
        rc, Po = oracle.cons_to_prim(kind, 0.9375, 0.3, X, GAM, Uo, P)
        bsq = oracle.state_at(kind, 0.9375, 0.3, X, P)["bsq"]
        cond = gam2 * (P[0] + P[1] + bsq) / P[1]
        assert rc == 0
        assert abs(out[0] - Po[0]) <= 64 * U53 * cond * gam2 * Po[0], it
        assert abs(out[1] - Po[1]) <= 64 * U53 * cond * gam2 * Po[1], it
        lv = np.sqrt(np.diag(gcov)[1:])
        assert np.abs((out[2:5] - Po[2:5]) * lv).max() <= 64 * U53 * gam2 * max(1.0, cond * P[1] / P[0]), it
        assert np.array_equal(out[5:8], Uo[5:8] * g[23])
        assert abs(bl[1] ** 2 - gam2) <= 64 * U53 * gam2 * cond


def test_unusual_input_is_left_to_the_caller(wide):
    """NaN, infinities, D <= 0, v^2 beyond 1 and negative u get no answer."""
    g = np.array([-1.0, 0, 0, 0, 1, 0, 0, 1, 0, 1] * 2 + [1.0, 1.0, 1.0, 1.0, 0.0])
    good = np.array([1.0, -2.0, 0.3, 0.0, 0.1, 0.2, 0.0, 0.1])  # U_u = -(energy) + rho
    out, bl = np.zeros(8), np.zeros(2)
    call = lambda U: wide.invert(_p(U), _p(g), ctypes.c_double(2.0), 1, _p(out), _p(bl))  # noqa: E731
    assert call(good) == 1
    for v, x in [(0, np.nan), (3, np.inf), (6, -np.inf), (0, 0.0), (0, -1.0), (2, 50.0), (1, 0.5)]:
        U = good.copy()
        U[v] = x
        assert call(U) == 0, (v, x)


@pytest.mark.gpu
@pytest.mark.parametrize("shear", ["block", "coupled"])
def test_uniform_state_stays_uniform(shear):
    """A uniform state in flat space in a sheared basis (with "coupled", one the
    library's own metrics never show the update) has no divergence and no
    source: two cycles return it, to the inversion's rounding."""
    import torch
    from paper_2110_10191_gb300 import grmhd, problems as pb
    from test_gpu_face_flux import SHEARS, _metric
    assert torch.cuda.is_available()
    pr = pb.linear_mode(8)
    pr.n = (9, 6, 5)
    P = np.zeros((8, 5, 6, 9))
    P[:] = np.array([0.7, 0.4, 0.3, -0.2, 0.5, 0.6, -0.1, 0.2])[:, None, None, None]
    sim = grmhd.Sim(pr)
    met = _metric(SHEARS[shear])
    for loc in range(3):
        geo = np.zeros((34,) + sim.s[1::-1])
        geo[:16], geo[16:32] = met[0].reshape(16)[:, None, None], met[1].reshape(16)[:, None, None]
        geo[32], geo[33] = met[2], met[3]
        sim.set_geom(loc, geo)
    sim.set_geom(3, np.zeros((64,) + sim.s[1::-1]))
    sim.set_prims(P)
    st = sim.step(2)
    assert st["t"] > 0.0 and st["inv_failures"] == 0
    # u is recovered from an energy of about ten times its size: 64 roundings of it
    assert np.abs(sim.get_prims() - P).max() <= 10 * 64 * U53
    sim.close()
