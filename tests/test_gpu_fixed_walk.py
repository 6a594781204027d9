"""The FP64 kernel walks a segment through the fluence grid in fixed point and
must still tally the oracle's integers: one and many voxels per axis, segments
along, almost along and on the planes, and scales from tiny to large."""
import math

import numpy as np
import pytest

import oracle as O
import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu


def _workload(n, tilt, scale, mu_s, npackets=400):
    # few scatterings: long segments; a beam on the planes x = 0 and y = 0 (n even)
    s = scale
    prims = (W.Prim(W.BOX, (0.0, 0.0, 0.0, 0.5 * s, 0.5 * s, 0.5 * s)),)
    regions = (W.Region(W.prim_program([0]), 0.2 / s, mu_s / s, 0.5, 1.2),)
    b = 0.6 * s
    norm = math.sqrt(1.0 + tilt * tilt)
    scene = W.Scene(prims, regions, 1.0, (-b, -b, -b), (b, b, b), delta=1e-5 * s)
    return W.Workload("walk", scene, W.Source(W.PENCIL, (0.0, 0.0, 0.55 * s), (tilt / norm, 0.0, -1.0 / norm)),
                      W.Grid((-0.5 * s, -0.5 * s, -0.5 * s), (0.5 * s, 0.5 * s, 0.5 * s), n), npackets, 21,
                      "fp64").with_stepping(W.SEGMENT)


CASES = [((1, 1, 1), 0.0, 1.0, 3.0), ((64, 64, 64), 0.0, 1.0, 3.0), ((64, 64, 64), 0.3, 1.0, 0.0),
         ((64, 48, 32), 1e-6, 1.0, 1.0), ((64, 48, 32), 1e-9, 1.0, 1.0), ((64, 48, 32), 1e-13, 1.0, 1.0),
         ((333, 1, 77), 0.1, 1.0, 3.0), ((2, 500, 500), 0.7, 1.0, 1.0), ((63, 65, 67), 1.0, 1.0, 10.0),
         ((80, 80, 80), 0.2, 1e-4, 3.0), ((80, 80, 80), 0.2, 1e3, 3.0), ((80, 80, 80), 0.2, 1e6, 3.0)]


@pytest.mark.parametrize("n,tilt,scale,mu_s", CASES)
def test_walk_equals_oracle(n, tilt, scale, mu_s):
    import torch
    ctx = smc.Context(0)
    wl = _workload(n, tilt, scale, mu_s)
    fo, to = O.run(wl)[:2]
    plan = ctx.plan(wl, "fp64")
    flu = torch.zeros((n[2], n[1], n[0]), dtype=torch.int64, device="cuda")
    tot = smc.totals_tensor()
    plan.launch(0, wl.npackets, wl.seed, flu, tot)
    torch.cuda.synchronize()
    assert plan.status() == 0
    plan.close()
    ctx.close()
    t = smc.totals_from_tensor(tot)
    for k in ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps"):
        assert t[k] == to[k], k
    assert np.array_equal(flu.cpu().numpy(), fo)
