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


@pytest.mark.parametrize("make,precision,n", [
    (W.three_layer_slab, "mixed", (3 << 18) - 1), (W.three_layer_slab, "mixed", 3 << 18),
    (lambda: W.iso_sphere(10.0), "mixed", (5 << 14) - 1), (lambda: W.iso_sphere(10.0), "mixed", 5 << 14),
    (W.vessel_network, "mixed", 20_000), (W.sdf_gallery, "mixed", 5_000),
    (W.glass_sphere_beam, "fp64", (1 << 19) - 1), (W.glass_sphere_beam, "fp64", 1 << 19)])
def test_default_shape_same_results(make, precision, n):
    """Both sides of the sizes at which the default launch shape changes, and
    the scenes with a default of their own: the same tallies as every chosen
    variant's."""
    import torch
    ctx = smc.Context(0)
    wl = make().with_packets(n).with_stepping(W.SEGMENT)
    got = []
    for variant in (None, 0, 1, 2):
        plan = ctx.plan(wl, precision)
        if variant is not None:
            plan.set_variant(variant)
        flu = torch.zeros(wl.grid.size, dtype=torch.int64, device="cuda")
        tot = smc.totals_tensor()
        plan.launch(0, n, 5, flu, tot)
        torch.cuda.synchronize()
        assert plan.status() == 0
        plan.close()
        got.append((flu, tot[:14].clone()))
    ctx.close()
    assert int(got[0][1][5]) == n
    for flu, tot in got[1:]:
        assert torch.equal(flu, got[0][0]) and torch.equal(tot, got[0][1])
