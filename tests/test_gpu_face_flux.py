"""The face fluxes against a plain numpy reference in extended precision, at the
edges of the kernel's layout (two lanes per face, 16 faces per warp) and for a
loaded metric that couples X2 to the other coordinates, which the library's own
metrics do not and for which the kernel takes its general path.

The metrics are constant, flat space in a sheared basis, so that the state at
every face is exact data.  Tolerance: the flux tolerance of the parity tests,
1e-12 of the largest flux of its group; each flux is a sum of at most a dozen
products rounded to 2^-53, whose largest is below ten times that scale."""
import numpy as np
import pytest

from paper_2110_10191_gb300 import problems as pb

pytestmark = pytest.mark.gpu


def _metric(shear):
    """(g_mn, g^mn, sqrt(-g), lapse) of flat space in the basis dx -> (1 + S) dx."""
    J = np.eye(4, dtype=np.longdouble)
    for (a, b), v in shear.items():
        J[a, b] = v
    eta = np.diag([-1.0, 1.0, 1.0, 1.0]).astype(np.longdouble)
    g = (J.T @ eta @ J).astype(np.float64)
    gi = np.linalg.inv(g)
    gi = (gi + gi.T) / 2
    return g, gi, np.sqrt(-np.linalg.det(g)), 1.0 / np.sqrt(-gi[0, 0])


def _mc(P, ax):
    a, c, e = np.roll(P, 1, ax), P, np.roll(P, -1, ax)
    dm, dp = c - a, e - c
    m = np.minimum(np.minimum(2 * abs(dm), 2 * abs(dp)), abs(dm + dp) / 2)
    h = np.where(dm * dp > 0, np.sign(dm) * m, 0) / 2
    return c - h, c + h


def _state(P, met, gam, d):
    g, gi, gdet, al = met
    v, B = P[2:5], P[5:8]
    low = [sum(g[i + 1, j + 1] * v[j] for j in range(3)) for i in range(3)]
    gm = np.sqrt(1 + sum(low[i] * v[i] for i in range(3)))
    u = [gm / al] + [v[i] - gm * al * gi[0, i + 1] for i in range(3)]
    ul = [sum(g[m, n] * u[n] for n in range(4)) for m in range(4)]
    bt = sum(B[i] * ul[i + 1] for i in range(3))
    b = [bt] + [(B[i] + bt * u[i + 1]) / u[0] for i in range(3)]
    bl = [sum(g[m, n] * b[n] for n in range(4)) for m in range(4)]
    b2 = sum(b[m] * bl[m] for m in range(4))
    pg = (gam - 1) * P[1]
    w, pt = P[0] + P[1] + pg + b2, pg + b2 / 2

    def rows(k):
        T = [w * u[k] * ul[n] - b[k] * bl[n] + (pt if n == k else 0) for n in range(4)]
        return np.stack([P[0] * u[k], T[0] + P[0] * u[k], T[1], T[2], T[3]] +
                        [b[i] * u[k] - b[k] * u[i] for i in (1, 2, 3)]) * gdet
    c2 = (gam * pg + b2) / w
    qa = u[0] ** 2 - (gi[0, 0] + u[0] ** 2) * c2
    hb = u[d] * u[0] - (gi[0, d] + u[d] * u[0]) * c2
    qc = u[d] ** 2 - (gi[d, d] + u[d] ** 2) * c2
    root = np.sqrt(np.maximum(hb * hb - qa * qc, 0))
    return rows(d), rows(0), np.maximum(abs((hb + root) / qa), abs((hb - root) / qa))


SHEARS = {
    "flat": {},
    "block": {(0, 1): 0.2, (1, 1): 1.5, (1, 3): 0.3, (0, 3): -0.1, (2, 2): 0.7},
    "coupled": {(0, 1): 0.2, (0, 2): 0.15, (1, 2): -0.4, (2, 3): 0.25, (1, 3): 0.3, (3, 3): 2.0},
}


@pytest.mark.parametrize("shear", sorted(SHEARS))
@pytest.mark.parametrize("n", [(4, 5, 3), (13, 4, 6), (17, 16, 4), (31, 7, 1)])
def test_face_fluxes(shear, n):
    import torch
    from paper_2110_10191_gb300 import grmhd
    assert torch.cuda.is_available()
    rng = np.random.default_rng(sum(n))
    pr = pb.linear_mode(8, recon=pb.RECON_MC)
    pr.n, pr.xmax = n, (1.0, 1.0, 1.0)
    P = np.zeros((8,) + n[::-1])
    P[0] = np.exp(rng.normal(size=P[0].shape))
    P[1] = P[0] * np.exp(rng.normal(size=P[0].shape) - 2)
    P[2:5] = 0.7 * rng.normal(size=P[2:5].shape)
    P[5:8] = rng.normal(size=P[5:8].shape)
    met = _metric(SHEARS[shear])
    sim = grmhd.Sim(pr)
    for loc in range(3):
        geo = np.zeros((34,) + sim.s[1::-1])
        geo[:16] = met[0].reshape(16)[:, None, None]
        geo[16:32] = met[1].reshape(16)[:, None, None]
        geo[32], geo[33] = met[2], met[3]
        sim.set_geom(loc, geo)
    sim.set_prims(P)
    F, ct = sim.fluxes()
    sim.close()
    met = tuple(np.asarray(m, dtype=np.longdouble) for m in met)
    Pl = P.astype(np.longdouble)
    for d in (1, 2, 3):
        lo, hi = _mc(Pl, 4 - d)
        FL, UL, cL = _state(np.roll(hi, 1, 4 - d), met, pr.gamma, d)
        FR, UR, cR = _state(lo, met, pr.gamma, d)
        c = np.maximum(cL, cR)
        want = 0.5 * (FL + FR - c * (UR - UL))
        assert abs(ct[d - 1] - c.max()) <= 1e-12 * c.max()
        got = F[d - 1][:, 3:-3, 3:-3, 3:-3]  # faces below the interior zones, before flux-CT's rows
        scale = np.abs(want[:5]).max()
        assert np.abs(got[:5] - want[:5]).max() <= 1e-12 * scale, (d, shear)
