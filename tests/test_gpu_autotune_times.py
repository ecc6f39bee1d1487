"""grmhd_autotune's ms_before is one pass of each tuned kernel, each counted once."""
import pytest

from paper_2110_10191_gb300 import problems as pb

pytestmark = pytest.mark.gpu


def test_each_kernel_is_counted_once():
    """FP32 fluxes, where the update's source pass is a third of the tuned time: no more
    than the same kernels take in a step's own profile (half a cycle; 15% for the
    caches' state and the clock)."""
    import torch

    from paper_2110_10191_gb300 import grmhd
    assert torch.cuda.is_available()
    pr = pb.fm_torus(96, 96, 96)
    pr.precision = grmhd.PREC_MIXED
    with grmhd.Sim(pr) as s:
        s.set_prims(pr.P)
        s.step(10)
        s.profile(True)
        s.step(2)
        s.get_profile(reset=True)
        s.step(10)
        t = s.get_profile(reset=True)
        s.profile(False)
        per_stage = sum(t[k][0] for k in ("recon", "flux", "update")) / 20
        before, _ = s.autotune(trials=20)
    assert before <= 1.15 * per_stage
