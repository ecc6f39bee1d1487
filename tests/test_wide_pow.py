"""log2, 2^y and Kawazura's heating share in Wide numbers (csrc/wide_pow.cuh), built for
the host, against numpy's extended precision.

Tolerances: the logarithm's table entry and its last product are truncated at 2^-55
each, its series below 2^-58: 2^-54 absolute.  2^y truncates y at 2^-55 (relative
error ln 2 times that) and is then rounded to a double, 2^-53: together below 2^-52.
The extended type's own log2 and exp2 are good to 2^-63 of values below 2^8.  The share:
a dozen operations and constants at 2^-53 on u - u_e, whose condition is (u + u_e)/|u -
u_e|, and on the exponent, at most 100 where the share depends on it: 2^-50 times both."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2110_10191_gb300 import build as _build

SRC = r"""
#include "wide_pow.cuh"
using namespace grmhd;
extern "C" void logs(long n, const double *x, long long *l) {
  for (long i = 0; i < n; i++) l[i] = w_log2(wide(x[i]));
}
extern "C" void exps(long n, const double *y, double *e) {
  for (long i = 0; i < n; i++) {
    Wide w = wide(y[i]);
    w.m >>= 1;
    w.x += 1;
    e[i] = w_to_double(w_exp2(w));
  }
}
extern "C" void shares(long n, double game, double gamp, const double *rho, const double *u,
                       const double *kel, const double *bsq, double *f) {
  for (long i = 0; i < n; i++)
    f[i] = w_to_double(wide_kawazura(game, gamp, 1.0 / (game - 1.0), rho[i],
                                     w_log_num(w_log2(wide(rho[i]))), u[i], kel[i], bsq[i]));
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("pow")
    (d / "w.cu").write_text(SRC)
    so = str(d / "w.so")
    subprocess.run([_build.nvcc(), "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", _build.CSRC, "-o", so, str(d / "w.cu")], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return ctypes.c_void_p(a.ctypes.data)


def test_log2(lib):
    rng = np.random.default_rng(1)
    edge = 1 + np.arange(64) / 64.0  # the table's intervals, from both sides
    x = np.concatenate([np.exp(rng.uniform(-60, 60, 20000)), 1 + rng.normal(size=2000) * 1e-9,
                        edge, np.nextafter(edge, 0), np.nextafter(edge, 4), [2.0 ** -249, 2.0 ** 249]])
    l = np.zeros(x.size, dtype=np.int64)
    lib.logs(ctypes.c_long(x.size), _p(x), _p(l))
    got = l.astype(np.longdouble) / np.longdouble(2) ** 55
    assert np.abs(got - np.log2(x.astype(np.longdouble))).max() <= 2.0 ** -54


def test_exp2(lib):
    rng = np.random.default_rng(2)
    edge = np.arange(-128, 129) / 64.0
    y = np.concatenate([rng.uniform(-127, 127, 20000), rng.normal(size=2000) * 1e-6, edge,
                        np.nextafter(edge, -9), np.nextafter(edge, 9), [0.0, -0.0, 127.99, -127.99]])
    e = np.zeros(y.size)
    lib.exps(ctypes.c_long(y.size), _p(y), _p(e))
    want = np.exp2(y.astype(np.longdouble))
    assert (np.abs(e - want) / want).max() <= 2.0 ** -52
    far = np.array([-256.0, -1e3, -1e19, -1e300])
    lib.exps(ctypes.c_long(far.size), _p(far), _p(e))
    assert (e[:far.size] == 0).all()


@pytest.mark.parametrize("game,gamp", [(4.0 / 3.0, 5.0 / 3.0), (1.4, 4.0 / 3.0)])
def test_kawazura_share(lib, game, gamp):
    rng = np.random.default_rng(3)
    n = 20000
    rho = np.exp(rng.uniform(-30, 5, n))
    u = rho * np.exp(rng.uniform(-12, 3, n))
    kel = (game - 1) * u * rho ** -game * rng.choice([1.0, 0.5, 1e-1, 1e-3, 1e-8, 3.0], n)
    bsq = u * np.exp(rng.uniform(-20, 10, n))
    bsq[::7], bsq[1::7], bsq[2::7] = 0.0, 1e-300, 5e-324  # none, and what rounding leaves
    f = np.zeros(n)
    lib.shares(ctypes.c_long(n), ctypes.c_double(game), ctypes.c_double(gamp), _p(rho), _p(u),
               _p(kel), _p(bsq), _p(f))
    r, w, k, b = (q.astype(np.longdouble) for q in (rho, u, kel, bsq))
    e1, p1 = np.longdouble(game - 1.0), np.longdouble(gamp - 1.0)
    Te = k * r ** e1
    ue = Te * r / e1
    Tp = np.abs(p1 * (w - ue) / r)
    with np.errstate(divide="ignore", over="ignore"):
        trat = np.clip(Tp / Te, 1e-20, 1e20)
        beta = np.clip(np.where(b > 0, 2 * r * Tp / b, 1e20), 1e-20, 1e20)
        x = np.longdouble("0.1") / trat
        want = 1 / (1 + 35 / (1 + (beta / 15) ** np.longdouble(-1.4) * np.exp(-x)))
        cond = (1 + (w + ue) / np.abs(w - ue)) * (1 + np.minimum(x, 100))
    assert (np.abs(f - want) / want <= 2.0 ** -50 * cond).all()
