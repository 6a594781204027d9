"""The launch without allocation at the largest scene that its scratch takes:
128 primitives, 16 regions, an unused frame, and 1024 planes on an axis.  FP64
tallies are those of a plan launch and of the oracle."""
import ctypes as C

import numpy as np
import pytest

import oracle as O
import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu


def _largest(n, soft):
    """Sixteen regions of eight blended spheres (soft: one of them of 100, the others single)."""
    rng = np.random.Generator(np.random.PCG64(12))
    prims = tuple(W.Prim(W.SPHERE, tuple(float(v) for v in (*rng.uniform(-0.8, 0.8, 3), rng.uniform(0.1, 0.3))))
                  for _ in range(128))
    parts = [range(8 * r, 8 * r + 8) for r in range(16)]
    if soft:
        parts = [range(r, r + 1) for r in range(15)] + [range(15, 115)]
    regions = tuple(W.Region(W.prim_program(list(p), W.SMOOTH_UNION, 0.01), 0.5, 8.0, 0.7, 1.3 + 0.01 * r)
                    for r, p in enumerate(parts))
    scene = W.Scene(prims, regions, 1.0, (-1.2, -1.2, -1.2), (1.2, 1.2, 1.2), stepping=W.SEGMENT)
    return W.Workload("largest", scene, W.Source(W.SQUARE, (0.0, 0.0, 1.1), (0.0, 0.0, -1.0), 0.9),
                      W.Grid((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0), n), 600, 9, "fp64")


@pytest.mark.parametrize("n", [(1024, 1024, 4), (4, 1024, 1024), (1024, 1, 1024)])
@pytest.mark.parametrize("soft", [False, True])
def test_largest_scene_without_allocation(n, soft):
    import torch
    wl = _largest(n, soft)
    fo, to, _ = O.run(wl, threads=4)
    ctx = smc.Context(0)
    plan = ctx.plan(wl, "fp64")
    flu = [torch.zeros(n[::-1], dtype=torch.int64, device="cuda") for _ in range(2)]
    tot = [smc.totals_tensor() for _ in range(2)]
    plan.launch(0, wl.npackets, wl.seed, flu[0], tot[0])
    m = smc.Marshalled(wl.scene, wl.source, wl.grid)
    X = m.xforms[0]                          # a frame that no primitive uses
    X.rot[:] = [1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0]
    X.s = 1.0
    m.scene.nxforms = 1
    rc = smc.lib().smcrt_run_noalloc(C.byref(m.scene), C.byref(m.source), C.byref(m.grid), 0, wl.npackets, wl.seed,
                                     0, flu[1].data_ptr(), tot[1].data_ptr(), None)
    torch.cuda.synchronize()
    assert rc == smc.OK and plan.status() == 0
    plan.close()
    ctx.close()
    assert torch.equal(flu[0], flu[1]) and torch.equal(tot[0][:14], tot[1][:14])
    assert np.array_equal(flu[0].cpu().numpy(), fo)
    t = smc.totals_from_tensor(tot[0])
    for k in ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps", "pieces"):
        assert t[k] == to[k], k
