"""Small plan launches spread their packets over all warps; how many lanes of
a warp carry packets must not change any result."""
import pytest

import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 63, 64, 65, 255, 256, 300])
def test_spread_over_warps(precision, n):
    """8 warps: one packet, fewer than warps, both sides of one and of eight
    lanes per warp, and more packets than lanes, against id blocks of 37."""
    import torch
    ctx = smc.Context(0)
    wl = W.glass_container(n, grid_n=16).with_stepping(W.SEGMENT)
    plan = ctx.plan(wl, precision)
    plan.set_launch(2, 128)
    got = []
    for block in (n, 37):
        flu = torch.zeros(wl.grid.size, dtype=torch.int64, device="cuda")
        tot = smc.totals_tensor()
        for b in range(0, n, block):
            plan.launch(b, min(block, n - b), 11, flu, tot)
        torch.cuda.synchronize()
        got.append((flu, tot[:14].clone()))
    assert plan.status() == 0
    assert int(got[0][1][5]) == n
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    plan.close()
    ctx.close()
