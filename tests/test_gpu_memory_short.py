"""Where the arrays that let a small grid's directions run side by side do not fit, the
grid is created without them and steps to the same result, bit for bit."""
import numpy as np
import pytest

from paper_2110_10191_gb300 import problems as pb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def grmhd():
    import torch

    from paper_2110_10191_gb300 import grmhd as m
    assert torch.cuda.is_available()
    return m


def _alone(grmhd, pr, steps):
    with grmhd.Sim(pr) as s:
        s.set_prims(pr.P)
        s.step(steps)
        return s.get_prims()


def _split_bytes(pr):
    n1, n2, n3 = pr.n
    return 5 * 8 * 8 * (n1 + 6) * (n2 + 6) * (n3 + 6)


def test_create_with_little_memory_free(grmhd):
    import torch
    pr = pb.fm_torus(96, 96, 96)
    ref = _alone(grmhd, pr, 2)  # (the kernels' local memory is held from here on)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - grmhd.footprint(pr) + _split_bytes(pr) // 2, dtype=torch.uint8,
                       device="cuda")
    try:
        got = _alone(grmhd, pr, 2)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(got, ref)


def test_server_budget_below_the_full_footprint(grmhd):
    pr = pb.fm_torus(24, 20, 8)
    ref = _alone(grmhd, pr, 3)
    srv = grmhd.Server(hbm_budget=grmhd.footprint(pr) - 1)
    try:
        srv.submit(0, pr, 3)
        srv.drain(timeout_ms=60000)
        res, st = srv.poll(4), srv.stats()
        assert len(res) == 1 and res[0]["status"] == 0 and np.array_equal(res[0]["P"], ref)
        assert st["peak_bytes"] == grmhd.footprint(pr) - _split_bytes(pr)
    finally:
        srv.close()
    srv = grmhd.Server(hbm_budget=grmhd.footprint(pr) - _split_bytes(pr) - 1)
    with pytest.raises(grmhd.GrmhdError):
        srv.submit(0, pr, 3)
    srv.close()


def test_blocks_of_a_large_grid_take_no_more_than_it(grmhd):
    """A decomposed grid of more than 2^21 zones does not run its directions side by
    side, whatever the size of its blocks."""
    import torch
    pr = pb.fm_torus(160, 128, 128)
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    d = grmhd.Decomp(pr, (2, 1, 1))
    used = free - torch.cuda.mem_get_info()[0]
    d.close()
    # ghosts of two blocks against one: 6 of 166 layers, and the exchange's tables
    assert used <= 1.1 * grmhd.footprint(pr)
