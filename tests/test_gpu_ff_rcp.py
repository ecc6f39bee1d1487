"""The float pairs' reciprocal and reciprocal square root (csrc/ff.cuh) on the device.

Bounds, relative.  1/a: the hardware's seed is within an ulp, 2^-23, so that e = 1 - a r is
below 1.5 x 2^-23 with a's low word; e's two roundings, that of e + e^2 and that of the
product each leave 2^-24 of that: 6 x 2^-47.  1/sqrt(a): the seed is within 2^-22.9, e = 1 -
a y^2 below 2^-21.8 with the low word; of its three roundings half enters, of e/2 + 3e^2/8
and the product one each, relative to e/2: (1.5 + 1) 2^-24 2^-21.8 = 2.5 x 2^-45.8."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2110_10191_gb300 import build as _build

pytestmark = pytest.mark.gpu
SRC = r"""
#include "ff.cuh"
using namespace grmhd;
__global__ void k(const float *hi, const float *lo, float *out, int n, int root) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const ff a = {hi[t], lo[t]}, r = root ? ff_rsqrt(a) : ff_rcp(a);
  out[t] = r.hi;
  out[n + t] = r.lo;
}
extern "C" int run(const float *hi, const float *lo, float *out, int n, int root) {
  k<<<(n + 255) / 256, 256>>>(hi, lo, out, n, root);
  return cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("root,bound", [(0, 6 * 2.0 ** -47), (1, 2.5 * 2.0 ** -45.8)])
def test_reciprocals(tmp_path, root, bound):
    import torch
    assert torch.cuda.is_available()
    (tmp_path / "r.cu").write_text(SRC)
    so = str(tmp_path / "r.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", _build.CSRC, "-o", so,
                    str(tmp_path / "r.cu")], check=True)
    rng = np.random.default_rng(2)
    n = 1 << 20
    x = 2.0 ** rng.uniform(-30, 30, n)
    x[:4096] = 2.0 ** rng.integers(-30, 30, 4096) * (1 + rng.integers(-4, 5, 4096) * 2.0 ** -22)
    hi = x.astype(np.float32)
    lo = (x - hi).astype(np.float32)
    d = [torch.from_numpy(q).cuda() for q in (hi, lo)] + [torch.zeros(2 * n, device="cuda")]
    p = [ctypes.c_void_p(q.data_ptr()) for q in d]
    assert ctypes.CDLL(so).run(*p, n, root) == 0
    r = d[2].cpu().numpy().astype(np.float64)
    a = hi.astype(np.float64) + lo  # exact
    ref = 1 / np.sqrt(a) if root else 1 / a
    # (the reference's own roundings: 2^-52)
    assert np.abs((r[:n] + r[n:]) / ref - 1).max() <= bound + 2.0 ** -51
