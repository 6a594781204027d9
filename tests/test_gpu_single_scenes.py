"""Scenes of simple regions run kernel instantiations that leave out what they
cannot need: every region one box (both precisions), one primitive (FP64), or
one box or a fold of capsules (a tree, FP64 here).  The same scene with one
region written as the union of its primitive with itself runs the plain
ones, whose arithmetic is the same, so every tally must be equal."""
import numpy as np
import pytest

import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu

# boxes: centre and half extents; spheres: centre and radius; capsules: ends and radius
SCENES = {
    "one": [(0.0, 0.0, 0.0, 0.5, 0.4, 0.3)],
    "layers": [(0.0, 0.0, 0.45, 4.0, 4.0, 0.05), (0.0, 0.0, 0.2, 4.0, 4.0, 0.2), (0.0, 0.0, -0.3, 4.0, 4.0, 0.3)],
    "nested": [(0.0, 0.0, 0.0, 0.5, 0.5, 0.5), (0.1, -0.1, 0.0, 0.3, 0.2, 0.25), (0.1, -0.1, 0.05, 0.1, 0.1, 0.1)],
    "edges": [(-0.2, 0.0, 0.0, 0.2, 0.5, 0.5), (0.2, 0.2, 0.0, 0.2, 0.3, 0.5), (0.2, -0.3, 0.0, 0.2, 0.2, 0.5),
              (0.0, 0.0, 0.0, 0.01, 0.01, 0.6)],
    "many": [(0.2 * (i % 4) - 0.3, 0.2 * (i // 4 % 4) - 0.3, 0.25 * (i // 16) - 0.2, 0.07, 0.08, 0.09)
             for i in range(16)],
    "sphere": [(0.0, 0.0, 0.0, 0.5)],
    "inclusions": [(0.0, 0.0, 0.0, 0.5, 0.5, 0.5), (0.1, 0.1, 0.1, 0.3), (-0.3, -0.2, -0.4, 0.2, 0.3, 0.4, 0.08),
                   (0.0, 0.0, -0.2, 0.2, 0.2, 0.05), (0.1, 0.1, 0.1, 0.25)],
}
# a box and a fold of capsules: how many, smoothing length (0: plain union)
TREES = {"tree2": (2, 0.0), "tree5": (5, 0.02), "tree12": (12, 0.0), "tree40": (40, 0.01)}


def _tree(name):
    rng = np.random.Generator(np.random.PCG64([11, TREES[name][0]]))
    caps = []
    for _ in range(TREES[name][0]):
        a = rng.uniform(-0.4, 0.4, 3)
        caps.append((*a, *(a + rng.uniform(-0.15, 0.15, 3)), rng.uniform(0.02, 0.06)))
    return [(0.0, 0.0, 0.0, 0.5, 0.5, 0.5), *caps]


def _workload(name, doubled, stepping):
    kinds = {4: W.SPHERE, 6: W.BOX, 7: W.CAPSULE}
    prims = tuple(W.Prim(kinds[len(b)], tuple(float(v) for v in b)) for b in SCENES.get(name) or _tree(name))
    regions = []
    if name in TREES:
        k = TREES[name][1]
        regions.append(W.Region(W.prim_program([0, 0] if doubled else [0]), 0.3, 5.0, 0.8, 1.4))
        fold = list(range(1, len(prims)))
        regions.append(W.Region(W.prim_program(fold, W.SMOOTH_UNION, k) if k else W.prim_program(fold),
                                2.0, 30.0, 0.9, 1.33))
        prims_of_one = []
    else:
        prims_of_one = range(len(prims))
    for i in prims_of_one:
        prog = W.prim_program([0, 0]) if doubled and i == 0 else W.prim_program([i])
        regions.append(W.Region(prog, 0.3 + 0.1 * (i % 5), 5.0 + 10.0 * (i % 3), 0.8, (1.4, 1.33, 1.5)[i % 3]))
    b = 0.7
    scene = W.Scene(prims, tuple(regions), 1.0, (-b, -b, -b), (b, b, b))
    return W.Workload("singles", scene, W.Source(W.SQUARE, (0.0, 0.0, 0.65), (0.0, 0.0, -1.0), 0.5),
                      W.Grid((-0.5, -0.5, -0.5), (0.5, 0.5, 0.5), (17, 16, 15)), 20_000, 3,
                      "mixed").with_stepping(stepping)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("stepping", [W.SPHERE_TRACING, W.SEGMENT])
@pytest.mark.parametrize("name", [*SCENES, *TREES])
def test_single_scenes_equal_plain(name, stepping, precision):
    import torch
    ctx = smc.Context(0)
    got = []
    runs = [(True, True), (False, True), (False, False)]
    if precision == "mixed" and name == "tree40":
        runs.pop()   # a mixed plan's cell list (folds of 16 and more) bounds moves; the fixed scratch has none
    for doubled, alloc in runs:
        wl = _workload(name, doubled, stepping)
        flu = torch.zeros(wl.grid.size, dtype=torch.int64, device="cuda")
        tot = smc.totals_tensor()
        if alloc:
            plan = ctx.plan(wl, precision)
            plan.launch(0, wl.npackets, wl.seed, flu, tot)
            torch.cuda.synchronize()
            assert plan.status() == 0
            plan.close()
        else:
            smc.run_noalloc(wl, 0, wl.npackets, wl.seed, flu, tot, precision)
            torch.cuda.synchronize()
        t = smc.totals_from_tensor(tot)
        got.append((flu, {k: t[k] for k in ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps")}))
    ctx.close()
    assert got[0][1]["packets"] == 20_000
    for flu, t in got[1:]:
        assert t == got[0][1]
        assert torch.equal(flu, got[0][0])
