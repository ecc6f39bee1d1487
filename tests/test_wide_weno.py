"""The WENO5 pair in 64-bit integer arithmetic (csrc/wide.cuh), built for the
host, against exact rational arithmetic.

Tolerance: a face value is c + corr with corr's weights and sums carried at 55
or more bits, so what rounds is the four first differences (half an ulp each,
in a candidate offset with coefficients of at most 7/6, and in the weights,
which move the value by less than the offsets' spread) and the last addition:
within 8 x 2^-53 of the stencil's largest magnitude."""
import ctypes
import itertools
import math
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2110_10191_gb300", "csrc")
U = 2.0 ** -53


@pytest.fixture(scope="module")
def pair(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")
    src = d / "w.cpp"
    src.write_text('#include "wide.cuh"\nextern "C" void pair(const double *x, double *o) {\n'
                   "  grmhd::weno5_wide_pair(x[0], x[1], x[2], x[3], x[4], o[0], o[1]);\n}\n")
    so = str(d / "w.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(src)],
                   check=True)
    L = ctypes.CDLL(so)

    def call(x):
        a, o = np.array(x, dtype=np.float64), np.zeros(2)
        L.pair(ctypes.c_void_p(a.ctypes.data), ctypes.c_void_p(o.ctypes.data))
        return float(o[0]), float(o[1])
    return call


def exact(x):
    a, b, c, d, e = (Fr(float(v)) for v in x)

    def hi(a, b, c, d, e):
        eps = Fr(1, 10 ** 26)
        be = [Fr(13, 12) * t * t + s * s / 4 for t, s in
              ((a - 2 * b + c, a - 4 * b + 3 * c), (b - 2 * c + d, b - d), (c - 2 * d + e, 3 * c - 4 * d + e))]
        w = [Fr(g, 10) / (eps + q) ** 2 for g, q in zip((1, 6, 3), be)]
        p = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
        return sum(u * v for u, v in zip(w, p)) / sum(w)
    return hi(e, d, c, b, a), hi(a, b, c, d, e)


def stencils(kind, rng, n=300):
    for _ in range(n):
        s = 10.0 ** rng.uniform(-24, 4)
        r = rng.uniform(-1, 1, 5)
        if kind == "rough":
            yield s * r
        elif kind == "smooth":
            yield s * (1 + 10.0 ** rng.uniform(-15, -1) * r)
        elif kind == "wave":
            yield s * (np.sin(rng.uniform(0, 7) + rng.uniform(0, 2) * np.arange(-2, 3)) + 3 * (r[0] > 0))
        elif kind == "decades":
            yield s * 10.0 ** (12 * r - 6) * np.sign(rng.uniform(-1, 1, 5))
        elif kind == "jump":  # one smooth side, the other 2 to 12 decades away, at each place
            k = rng.integers(1, 5)
            yield s * (1 + 0.1 * r) * np.where(np.arange(5) < k, 1.0, 10.0 ** rng.uniform(-12, -2))
        else:  # repeated values: differences that vanish
            yield s * rng.choice([0.0, 1.0, 1.0 + 2 ** -52, -1.0], 5)


@pytest.mark.parametrize("kind", ["rough", "smooth", "wave", "decades", "jump", "repeated"])
def test_pair_against_exact(pair, kind):
    for x in stencils(kind, np.random.default_rng(7)):
        got, want, big = pair(x), exact(x), float(np.abs(x).max())
        for g, w in zip(got, want):
            assert abs(Fr(g) - w) <= Fr(8 * U * big), (x, g, float(w))
        # a mirrored stencil swaps the two values, an opposite one turns them over
        assert pair(x[::-1]) == got[::-1]
        assert pair(-x) == (-got[0], -got[1])


def test_pair_special_values(pair):
    for c in (0.0, 3.0, -1e-300, 1e300):
        assert pair([c] * 5) == (c, c)
    for at, v in itertools.product(range(5), (math.nan, math.inf, -math.inf)):
        x = [1.0, 2.0, 4.0, 3.0, 1.5]
        x[at] = v
        assert all(math.isnan(y) for y in pair(x)), (at, v)
    tiny = np.array([1.0, 2.0, 3.0, 4.0, 5.0]) * 5e-324  # weights are the linear ones: 2.5, 3.5
    lo, hi = pair(tiny)
    assert {lo, hi} <= {2 * 5e-324, 3 * 5e-324, 4 * 5e-324} and lo <= hi
    lo, hi = pair(np.array([1.0, -1.0, 1.0, -1.0, 1.0]) * 1e300)  # FP64 weights would overflow
    assert abs(lo) <= 3e300 and abs(hi) <= 3e300
