"""Folds of many shapes run over cell lists in the mixed kernels, by a family
of instantiations of their own (plain scenes) or the general one, and by a
loop of their own where every listed shape is a capsule.  Each combination
must agree with the FP64 kernel, which has no cell lists."""
import numpy as np
import pytest

import bench
import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu

FX = 2.0 ** 32


def _fold(shapes, smooth, general, npackets):
    rng = np.random.Generator(np.random.PCG64([len(shapes), smooth, general]))
    prims = [W.Prim(W.BOX, (0.0, 0.0, 0.0, 0.5, 0.5, 0.5))]
    for i in range(26):
        c = [float(v) for v in rng.uniform(-0.4, 0.4, 3)]
        kind = shapes[i % len(shapes)]
        if kind == W.SPHERE:
            prims.append(W.Prim(kind, (*c, float(rng.uniform(0.03, 0.08)))))
        elif kind == W.BOX:
            prims.append(W.Prim(kind, (*c, *[float(v) for v in rng.uniform(0.02, 0.08, 3)])))
        else:
            e = [float(v + d) for v, d in zip(c, rng.uniform(-0.12, 0.12, 3))]
            prims.append(W.Prim(kind, (*c, *e, float(rng.uniform(0.02, 0.05)))))
    fold = list(range(1, 27))
    regions = [W.Region(W.prim_program([0]), 0.5, 20.0, 0.8, 1.33),
               W.Region(W.prim_program(fold, W.SMOOTH_UNION, 0.01) if smooth else W.prim_program(fold),
                        4.0, 40.0, 0.9, 1.4)]
    if general:
        prims.append(W.Prim(W.TORUS, (0.0, 0.0, 0.0, 0.2, 0.05)))
        regions.append(W.Region(W.prim_program([27]), 1.0, 10.0, 0.5, 1.5))
    b = 0.6
    scene = W.Scene(tuple(prims), tuple(regions), 1.0, (-b, -b, -b), (b, b, b))
    return W.Workload("fold", scene, W.Source(W.SQUARE, (0.0, 0.0, 0.55), (0.0, 0.0, -1.0), 0.4),
                      W.Grid((-0.5, -0.5, -0.5), (0.5, 0.5, 0.5), (16, 16, 16)), npackets, 7, "mixed")


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("smooth", [False, True])
@pytest.mark.parametrize("shapes", [(W.CAPSULE,), (W.CAPSULE, W.SPHERE), (W.SPHERE, W.BOX, W.CAPSULE), (W.BOX,)],
                         ids=lambda s: "+".join(s))
def test_cell_lists_match_fp64(shapes, smooth, general):
    """R, T and A of the two kernels on the same 50000 ids: 4 sigma of the
    paired differences (16 * 3 comparisons: one in 300 by chance); every
    packet's weight balances to the tally's rounding."""
    import torch
    ctx = smc.Context(0)
    wl = _fold(shapes, smooth, general, 50_000).with_stepping(W.SEGMENT)
    rec = {}
    for precision in ("mixed", "fp64"):
        plan = ctx.plan(wl, precision)
        tot = smc.totals_tensor()
        out = torch.zeros(wl.npackets * 8, dtype=torch.int64, device="cuda")
        plan.launch(0, wl.npackets, wl.seed, None, tot, out)
        torch.cuda.synchronize()
        assert plan.status() == 0
        assert smc.totals_from_tensor(tot)["max_steps_hit"] == 0
        plan.close()
        rec[precision] = out.cpu().numpy().view(smc.RECORD_DTYPE)
    ctx.close()
    for key in ("R", "T", "A"):
        z = bench.paired_z(rec["mixed"][key] / FX, rec["fp64"][key] / FX)
        assert abs(z) < 4.0, (key, z)
    r = rec["mixed"]
    assert np.all(np.abs((r["R"] + r["T"] + r["A"] + r["killed"] - r["gain"]) / FX - 1.0) < 1e-4)
