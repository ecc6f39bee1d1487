"""Reading the state between steps leaves the next step as it is: bit for bit, on grids
whose ghosts are set once and kept (fixed sides) and on a periodic one."""
import numpy as np
import pytest

from paper_2110_10191_gb300 import problems as pb

pytestmark = pytest.mark.gpu


def _problem(name):
    if name == "mode":
        return pb.linear_mode(16)
    pr = pb.bondi(32, 24, n3=2, recon=pb.RECON_WENO5)
    return pb.with_electrons(pr, model=pb.ELEC_WERNER) if name == "bondi_electrons" else pr


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("name", ["mode", "bondi", "bondi_electrons"])
def test_read_between_steps(name, on_device):
    import torch

    from paper_2110_10191_gb300 import grmhd
    assert torch.cuda.is_available()
    pr = _problem(name)
    with grmhd.Sim(pr) as a, grmhd.Sim(pr) as b:
        for sim in (a, b):
            sim.set_prims(pr.info.get("P_ghost", pr.P))
            if pr.electrons:
                sim.set_electrons(pr.info.get("K_ghost", pr.K))
        out = torch.empty(pr.P.shape, dtype=torch.float64, device="cuda") if on_device else None
        a.step(1)
        b.step(1)
        b.get_prims(out=out)
        if pr.electrons:
            b.get_electrons()
        a.step(1)
        b.step(1)
        assert np.array_equal(a.get_prims(True), b.get_prims(True))
        if pr.electrons:
            assert np.array_equal(a.get_electrons(True), b.get_electrons(True))
