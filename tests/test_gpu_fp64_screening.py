"""The FP64 kernel screens with FP32 which surfaces, planes and voxels count
and computes only those in FP64.  Its results must stay the oracle's, bit for
bit, on every form of scene it accepts: seeded scenes of folds, other CSG
programs, coincident faces, thin and touching shapes, coordinates far from
the origin, scales at and beyond the screening's range, and grids whose
planes do or do not meet the packets' paths."""
import math
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps")


def _prim(rng, lo, hi, size):
    c = [float(v) for v in rng.uniform(lo, hi, 3)]
    kind = int(rng.integers(3))
    if kind == 0:
        return W.Prim(W.SPHERE, (*c, float(rng.uniform(0.3, 1.0) * size)))
    if kind == 1:
        return W.Prim(W.BOX, (*c, *[float(v) for v in rng.uniform(0.2, 1.0, 3) * size]))
    d = rng.normal(size=3)
    d *= rng.uniform(0.3, 1.5) * size / np.linalg.norm(d)
    return W.Prim(W.CAPSULE, (*c, *[float(a + b) for a, b in zip(c, d)], float(rng.uniform(0.1, 0.5) * size)))


def _scene(form, seed):
    rng = np.random.Generator(np.random.PCG64([seed, len(form)]))
    off, scale = {"far": ((37.0, -81.0, 64.0), 1.0), "small": ((0.0, 0.0, 0.0), 1e-4),
                  "tiny": ((0.0, 0.0, 0.0), 1e-7)}.get(form, ((0.0, 0.0, 0.0), 1.0))
    prims, regions = [], []

    def region(program):
        mu_s, mu_a = float(rng.uniform(1.0, 30.0)), float(rng.uniform(0.05, 2.0))
        regions.append(W.Region(tuple(program), mu_a / scale, mu_s / scale, float(rng.uniform(0.0, 0.95)),
                                float(rng.choice([1.0, 1.33, 1.4, 1.5]))))

    def add(p):
        q = list(p.params)
        if p.kind == W.CAPSULE:
            q = [v * scale + off[k % 3] for k, v in enumerate(q[:6])] + [q[6] * scale]
        else:
            q = [v * scale + off[k] for k, v in enumerate(q[:3])] + [v * scale for v in q[3:]]
        prims.append(W.Prim(p.kind, tuple(q)))
        return len(prims) - 1

    if form == "layers":                     # coincident faces on grid planes
        z = 0.0
        for t in (0.1, 0.25, 0.5):
            region(W.prim_program([add(W.Prim(W.BOX, (0.0, 0.0, 0.5 - z - t / 2, 3.0, 3.0, t / 2)))]))
            z += t
    elif form == "thin":                     # sheets about as thin as the FP32 error bound
        region(W.prim_program([add(W.Prim(W.BOX, (0.0, 0.0, 0.0, 0.8, 0.8, 0.5)))]))
        for k in range(3):
            region(W.prim_program([add(W.Prim(W.BOX, (0.0, 0.0, -0.3 + 0.25 * k, 0.7, 0.7, 10.0 ** -(k + 3))))]))
    else:
        region(W.prim_program([add(W.Prim(W.BOX, (0.0, 0.0, 0.0, 0.9, 0.9, 0.8)))]))
        for _ in range(int(rng.integers(1, 4))):
            n = int(rng.integers(20, 70)) if form == "fold" else int(rng.integers(1, 6))
            ids = [add(_prim(rng, -0.7, 0.7, 0.15 if form == "fold" else 0.4)) for _ in range(n)]
            prog = [W.Node(W.PRIM, ids[0])]
            ops = ([W.UNION, W.SMOOTH_UNION] if form == "fold" else
                   [W.UNION, W.SMOOTH_UNION, W.INTERSECT, W.SUBTRACT])
            one = str(rng.choice(ops))
            for i in ids[1:]:
                op = one if rng.random() < 0.7 else str(rng.choice(ops))
                prog += [W.Node(W.PRIM, i), W.Node(op, -1, float(10.0 ** rng.uniform(-4, -1)) * scale)]
            if form == "csg" and n >= 4:     # a subtree of its own: binary operators over the stack
                prog = [W.Node(W.PRIM, ids[0]), W.Node(W.PRIM, ids[1]), W.Node(W.UNION),
                        W.Node(W.PRIM, ids[2]), W.Node(W.PRIM, ids[3]), W.Node(W.SMOOTH_UNION, -1, 0.02 * scale),
                        W.Node(W.SUBTRACT if rng.random() < 0.5 else W.INTERSECT)]
            region(prog)
    b = 1.25
    lo, hi = (tuple(s * b * scale + o for o in off) for s in (-1.0, 1.0))
    scene = W.Scene(tuple(prims), tuple(regions), 1.0, lo, hi, delta=1e-6 * scale, max_steps=20_000,
                    stepping=W.SEGMENT if seed % 2 == 0 else W.SPHERE_TRACING)
    pos = (off[0], off[1], off[2] + 1.1 * scale)
    src = [W.Source(W.PENCIL, pos, (0.0, 0.0, -1.0)),
           W.Source(W.SQUARE, pos, (0.0, 0.0, -1.0), 0.6 * scale),
           W.Source(W.DISC, pos, (math.sin(0.3), 0.0, -math.cos(0.3)), 0.5 * scale),
           W.Source(W.ISO_POINT, tuple(off), (0.0, 0.0, 1.0))][seed % 4]
    n = [(10, 10, 10), (7, 31, 1), (64, 50, 33)][seed % 3]
    g = [1.0, 0.5, 1.5][seed // 2 % 3]
    grid = W.Grid(tuple(o - g * scale for o in off), tuple(o + g * scale for o in off), n)
    return W.Workload(f"{form}{seed}", scene, src, grid, 120, 1000 + seed, "fp64")


@pytest.mark.parametrize("form", ["fold", "csg", "layers", "thin", "far", "small", "tiny"])
@pytest.mark.parametrize("seed", range(6))
def test_screened_fp64_is_the_oracles(form, seed):
    import torch
    wl = _scene(form, seed)
    fo, to, ro = O.run(wl, records=True)
    ctx = smc.Context(0)
    plan = ctx.plan(wl, "fp64")
    flu = torch.zeros(wl.grid.n[::-1], dtype=torch.int64, device="cuda")
    tot = smc.totals_tensor()
    rec = torch.zeros(wl.npackets * 8, dtype=torch.int64, device="cuda")
    plan.launch(0, wl.npackets, wl.seed, flu, tot, rec)
    torch.cuda.synchronize()
    assert plan.status() == 0
    tg = smc.totals_from_tensor(tot)
    for k in KEYS:
        assert tg[k] == to[k], (k, tg[k], to[k])
    assert np.array_equal(flu.cpu().numpy().reshape(-1), np.asarray(fo).reshape(-1))
    r = rec.cpu().numpy().view(smc.RECORD_DTYPE)
    for f in ("R", "T", "A", "killed", "gain", "scatters", "steps"):
        assert np.array_equal(r[f], ro[f]), f
    # the launch without allocation compiles its own copy of the tables
    if len(wl.scene.prims) <= 128 and len(wl.scene.regions) <= 16:
        f2, t2 = torch.zeros_like(flu), smc.totals_tensor()
        try:
            smc.run_noalloc(wl, 0, wl.npackets, wl.seed, f2, t2)
        except smc.SmcrtError as e:
            assert e.code == smc.ERR_NO_MEMORY
        else:
            torch.cuda.synchronize()
            assert torch.equal(f2, flu) and torch.equal(t2[:14], tot[:14])
    plan.close()
    ctx.close()
