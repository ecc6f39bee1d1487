"""The ghost fill in one pass against the three passes it stands for (X1 on the
interior rows, X2 on every i, X3 on every zone), written out in numpy: every kind
of boundary, fixed ghosts in each direction, directions shorter than the ghost
layer and of one zone.  Copies, sign changes and one IEEE product: equal bit for
bit."""
import numpy as np
import pytest

from paper_2110_10191_gb300 import problems as pb

pytestmark = pytest.mark.gpu
G = 3
PER, OUT, POL, FIX = (pb.BC_PERIODIC,) * 2, (pb.BC_OUTFLOW,) * 2, (pb.BC_POLAR,) * 2, (pb.BC_FIXED,) * 2


def _three_passes(P, K, n, bc, gdet):
    """P [8][k][j][i] and K [2][k][j][i] with their ghosts filled, pass by pass."""
    for ax, d in ((3, 0), (2, 1), (1, 2)):
        inner = [slice(None), slice(None), slice(None), slice(None)]
        if d < 2:
            inner[1] = slice(G, n[2] + G)
        if d < 1:
            inner[2] = slice(G, n[1] + G)
        for side in (0, 1):
            kind = bc[d][side]
            for g in range(G):
                dst = n[d] + G + g if side else g
                edge = n[d] + G - 1 if side else G
                src = {pb.BC_PERIODIC: (dst - G) % n[d] + G, pb.BC_OUTFLOW: edge,
                       pb.BC_POLAR: 2 * (n[d] + G) - 1 - dst if side else 2 * G - 1 - dst,
                       pb.BC_FIXED: dst}[kind]
                a, b = list(inner), list(inner)
                a[ax], b[ax] = dst, src
                a, b = tuple(a), tuple(b)
                P[a], K[a] = P[b], K[b]
                if kind == pb.BC_OUTFLOW:
                    P[a][5:8] *= gdet[None, None, G:n[1] + G, src] / gdet[None, None, G:n[1] + G, dst]
                    u1 = P[a][2]
                    u1[(u1 < 0) if side else (u1 > 0)] = 0.0
                if kind == pb.BC_POLAR:
                    P[a][[3, 6]] = -P[a][[3, 6]]
    return P, K


@pytest.mark.parametrize("n,bc", [((9, 5, 4), (OUT, POL, PER)), ((1, 2, 1), (PER, PER, PER)),
                                  ((7, 3, 1), (OUT, POL, PER)), ((5, 4, 2), (FIX, POL, PER)),
                                  ((4, 1, 5), (OUT, FIX, FIX)), ((2, 6, 3), (PER, FIX, PER)),
                                  ((6, 5, 7), ((pb.BC_FIXED, pb.BC_OUTFLOW),
                                               (pb.BC_FIXED, pb.BC_POLAR), FIX))])
def test_ghost_fill_is_the_three_passes(n, bc):
    import torch

    from paper_2110_10191_gb300 import grmhd
    assert torch.cuda.is_available()
    rng = np.random.default_rng(sum(n))
    pr = pb.linear_mode(8)
    pr.metric, pr.a, pr.hslope = pb.fm_torus(8, 8, 4).metric, 0.5, 0.3
    pr.xmin, pr.xmax, pr.n, pr.bc = (0.5, 0.0, 0.0), (3.0, 1.0, 6.0), n, bc
    s3 = tuple(q + 2 * G for q in n[::-1])
    P, K = np.abs(rng.normal(size=(8,) + s3)) + 0.1, np.abs(rng.normal(size=(2,) + s3)) + 0.1
    P[2:] *= rng.choice([-1.0, 1.0], size=P[2:].shape)
    pr.P = P[:, G:-G, G:-G, G:-G].copy()
    pr = pb.with_electrons(pr, pb.ELEC_CONSTANT, K=K[:, G:-G, G:-G, G:-G].copy())
    with grmhd.Sim(pr) as s:
        s.set_prims(P)
        s.set_electrons(K)
        got, gotK = s.get_prims(True), s.get_electrons(True)
        gdet = s.geom(0)[32]
    want, wantK = _three_passes(P.copy(), K.copy(), n, bc, gdet)
    assert np.array_equal(got, want)
    assert np.array_equal(gotK, wantK)
