"""Segment stepping in FP64 moves a packet as far as the oracle does, bit for
bit, in the scenes in which a bound of the move is easily lost: soft regions
(folds of more than eight smooth unions, which bound a move by their distance
alone) where the FP32 screening is off, and boxes with a margin, whose grown
shape has sharp corners nearer than the margin's distance."""
from dataclasses import replace

import numpy as np
import pytest
from test_gpu_fp64_screening import _scene

import oracle as O
import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("R", "T", "A", "killed", "gain", "packets", "scatters", "steps", "max_steps_hit")


def _check(wl, fluence=True):
    """Totals, records and (unless its units overflow) fluence of a plan launch and
    of the launch without allocation against the oracle's."""
    import torch
    fo, to, ro = O.run(wl, fluence=fluence, records=True)
    ctx = smc.Context(0)
    plan = ctx.plan(wl, "fp64")
    flu = torch.zeros(wl.grid.n[::-1], dtype=torch.int64, device="cuda") if fluence else None
    tot = smc.totals_tensor()
    rec = torch.zeros(wl.npackets * 8, dtype=torch.int64, device="cuda")
    plan.launch(0, wl.npackets, wl.seed, flu, tot, rec)
    f2, t2 = torch.zeros_like(flu) if fluence else None, smc.totals_tensor()
    smc.run_noalloc(wl, 0, wl.npackets, wl.seed, f2, t2)
    torch.cuda.synchronize()
    assert plan.status() == 0
    tg = smc.totals_from_tensor(tot)
    for k in KEYS + (("pieces",) if fluence else ()):
        assert tg[k] == to[k], (k, tg[k], to[k])
    r = rec.cpu().numpy().view(smc.RECORD_DTYPE)
    for f in ("R", "T", "A", "killed", "gain", "scatters", "steps"):
        assert np.array_equal(r[f], ro[f]), f
    assert torch.equal(t2[:14], tot[:14])
    if fluence:
        assert np.array_equal(flu.cpu().numpy().reshape(-1), np.asarray(fo).reshape(-1))
        assert torch.equal(f2, flu)
    plan.close()
    ctx.close()


def _scaled(wl, s):
    """The same scene in other units: lengths times s, coefficients over s."""
    prims = tuple(replace(p, params=tuple(v * s for v in p.params)) for p in wl.scene.prims)
    regions = tuple(replace(r, mu_a=r.mu_a / s, mu_s=r.mu_s / s,
                            program=tuple(replace(n, k=n.k * s) for n in r.program)) for r in wl.scene.regions)
    by = lambda v: tuple(x * s for x in v)
    scene = replace(wl.scene, prims=prims, regions=regions, delta=wl.scene.delta * s,
                    bbox_lo=by(wl.scene.bbox_lo), bbox_hi=by(wl.scene.bbox_hi))
    return replace(wl, scene=scene, source=replace(wl.source, pos=by(wl.source.pos), radius=wl.source.radius * s),
                   grid=replace(wl.grid, lo=by(wl.grid.lo), hi=by(wl.grid.hi)))


def _vessel(n=300):
    return W.vessel_network(n, precision="fp64", grid_n=20).with_stepping(W.SEGMENT)


def _wide(wl, half):
    """The tissue box (primitive 0) widened beyond the volume of interest."""
    p = wl.scene.prims[0].params
    box = W.Prim(W.BOX, p[:3] + (half, half, p[5]))
    return replace(wl, scene=replace(wl.scene, prims=(box,) + wl.scene.prims[1:]))


@pytest.mark.parametrize("scale", [1e-7, 1e-6, 1e13])
def test_soft_region_bounds_the_move_at_any_scale(scale):
    """(At 1e13 cm a track length overflows the fluence's units.)"""
    _check(_scaled(_vessel(), scale), fluence=scale < 1.0)


def test_soft_region_bounds_the_move_beside_a_wide_box():
    _check(_wide(_vessel(), 1e13))


@pytest.mark.parametrize("radius", [1e13, float("inf")])
def test_the_radius_of_a_pencil_changes_nothing(radius):
    wl = _vessel()
    _check(replace(wl, source=replace(wl.source, kind=W.PENCIL, radius=radius)))


def _blend(kinds, k, n, seed):
    """A smooth union of boxes (and spheres, capsules) with radius k in a
    scattering box; an odd seed puts a second, hard box beside it."""
    rng = np.random.Generator(np.random.PCG64(seed))
    prims = [W.Prim(W.BOX, (0.0, 0.0, 0.0, 1.0, 1.0, 1.0))]
    for kind in kinds:
        c = [float(v) for v in rng.uniform(-0.5, 0.5, 3)]
        if kind == W.BOX:
            prims.append(W.Prim(kind, (*c, *[float(v) for v in rng.uniform(0.1, 0.35, 3)])))
        elif kind == W.SPHERE:
            prims.append(W.Prim(kind, (*c, float(rng.uniform(0.15, 0.35)))))
        else:
            prims.append(W.Prim(kind, (*c, *[float(v) for v in rng.uniform(-0.5, 0.5, 3)], float(rng.uniform(0.05, 0.2)))))
    regions = [W.Region(W.prim_program([0]), 0.5, 10.0, 0.8, 1.33),
               W.Region(W.prim_program(list(range(1, len(prims))), W.SMOOTH_UNION, k), 1.0, 5.0, 0.7, 1.45)]
    if seed % 2:
        prims.append(W.Prim(W.BOX, (0.0, 0.0, -0.8, 0.3, 0.9, 0.1)))
        regions.append(W.Region(W.prim_program([len(prims) - 1]), 1.0, 20.0, 0.9, 1.5))
    scene = W.Scene(tuple(prims), tuple(regions), 1.0, (-1.2, -1.2, -1.2), (1.2, 1.2, 1.2), stepping=W.SEGMENT)
    return W.Workload("blend", scene, W.Source(W.SQUARE, (0.0, 0.0, 1.1), (0.0, 0.0, -1.0), 0.9),
                      W.Grid((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0), (21, 20, 19)), n, seed, "fp64")


BLENDS = [((W.BOX,) * 2, 0.2), ((W.BOX, W.SPHERE), 0.3), ((W.BOX,) * 8, 0.05), ((W.BOX,) * 4, 0.1),
          ((W.BOX, W.CAPSULE, W.BOX), 0.25), ((W.BOX, W.SPHERE, W.BOX, W.CAPSULE, W.BOX, W.BOX), 0.15)]


@pytest.mark.parametrize("kinds,k", BLENDS, ids=[f"{'+'.join(a)}-{k}" for a, k in BLENDS])
@pytest.mark.parametrize("seed", [1, 2])
def test_blended_boxes_move_as_the_oracle(kinds, k, seed):
    _check(_blend(kinds, k, 20_000, seed))


@pytest.mark.parametrize("seed", [230, 258, 332, 414, 562])
def test_folds_with_boxes_move_as_the_oracle(seed):
    _check(_scene("fold", seed))


def _boxes(seed, n=20_000):
    """Hard boxes with a coarse surface threshold: corners grown by delta / 2."""
    rng = np.random.Generator(np.random.PCG64([seed, 5]))
    prims = [W.Prim(W.BOX, (0.0, 0.0, 0.0, 1.0, 1.0, 1.0))]
    for _ in range(int(rng.integers(2, 9))):
        prims.append(W.Prim(W.BOX, tuple(float(v) for v in (*rng.uniform(-0.9, 0.9, 3), *rng.uniform(0.02, 0.4, 3)))))
    regions = tuple(W.Region(W.prim_program([i]), 0.3, float(rng.uniform(1.0, 20.0)), 0.8,
                             float(rng.choice([1.33, 1.4, 1.5]))) for i in range(len(prims)))
    scene = W.Scene(tuple(prims), regions, 1.0, (-1.2, -1.2, -1.2), (1.2, 1.2, 1.2), delta=float(rng.uniform(0.01, 0.05)),
                    max_steps=3000, stepping=W.SEGMENT)
    return W.Workload("boxes", scene, W.Source(W.SQUARE, (0.0, 0.0, 1.1), (0.0, 0.0, -1.0), 0.9),
                      W.Grid((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0), (21, 20, 19)), n, seed, "fp64")


@pytest.mark.parametrize("seed", [2, 10, 13, 173, 251, 284])
def test_hard_boxes_with_a_coarse_threshold_move_as_the_oracle(seed):
    _check(_boxes(seed))
