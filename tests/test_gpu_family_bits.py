"""The scene families of the mixed kernel give the same bits: a fold of
capsules with its cell list in the tree family, and, once a far-away region
that no packet comes near makes the scene none of its kind, in the culled one;
and served jobs, whose round takes the family that runs all its scenes, alone
and beside jobs that change the family."""
from dataclasses import replace

import numpy as np
import pytest

import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps", "scene_evals", "interfaces", "fresnel",
        "pieces", "max_steps_hit")


def _far(wl):
    """A union of two spheres 100 cm away: never the nearest surface."""
    n = len(wl.scene.prims)
    prims = wl.scene.prims + (W.Prim(W.SPHERE, (100.0, 0.0, 0.0, 0.5)), W.Prim(W.SPHERE, (100.4, 0.0, 0.0, 0.5)))
    regions = wl.scene.regions + (W.Region(W.prim_program([n, n + 1]), 1.0, 1.0, 0.5, 1.2),)
    return replace(wl, scene=replace(wl.scene, prims=prims, regions=regions))


@pytest.mark.parametrize("stepping", [W.SEGMENT, W.SPHERE_TRACING])
@pytest.mark.parametrize("smooth", [True, False])
def test_tree_and_culled_family_agree(smooth, stepping):
    ctx = smc.Context(0)
    wl = W.vessel_network(30_000, grid_n=50, smooth=smooth).with_stepping(stepping)
    want = ctx.run(wl, "mixed")
    got = ctx.run(_far(wl), "mixed")
    ctx.close()
    assert want[1]["packets"] == wl.npackets and want[1]["interfaces"] > 0
    for k in KEYS:
        assert got[1][k] == want[1][k], k
    assert np.array_equal(got[0], want[0])


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_served_beside_other_families(precision):
    """A plain and a vessel job: each alone, together, and beside the shape
    gallery."""
    n = 60_000 if precision == "mixed" else 4_000
    jobs = [W.glass_container(n, grid_n=32).with_stepping(W.SEGMENT),
            W.vessel_network(n, grid_n=40).with_stepping(W.SEGMENT)]
    gallery = W.sdf_gallery(5_000).with_stepping(W.SEGMENT)
    ctx = smc.Context(0)
    alone = [ctx.wait(ctx.submit(j, precision)) for j in jobs]
    for extra in ([], [gallery]):
        ids = [ctx.submit(j, precision) for j in jobs] + [ctx.submit(j, "mixed") for j in extra]
        got = [ctx.wait(i) for i in ids]
        for (flu, tot, _), (flu0, tot0, _) in zip(got, alone):
            assert np.array_equal(flu, flu0)
            for k in KEYS:
                assert tot[k] == tot0[k], k
    ctx.close()
