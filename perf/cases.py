"""What a user of the photon-packet library has it do, as measurable cases.

A case names a workload family (``workloads``), the call it goes through, the
precision, the step rule, the number of packets and the fluence grid.  The
calls are the library's public ones:

  launch   a plan kept by the program, launched on device tensors
           (fluence and totals zeroed, then accumulated into);
  records  the same with one record per packet;
  run      the synchronous one-shot call with a host fluence array;
  noalloc  the launch without device allocation;
  serve    several jobs submitted at once to a context that is already
           serving, and waited for.

Every output is a whole number (int64 fixed point and event counts).  The two
time statistics of the totals (busy cycles, parking events) depend on the
clock and are not results of a run, so the totals are given without them.
"""
import math
from dataclasses import replace

import numpy as np
import torch

import paper_2112_08035_gb300 as smc
import workloads as W

RESULTS = [f for f in smc.TOTAL_FIELDS if f not in ("busy_cycles", "parked")]
NRESULTS = len(RESULTS)          # the first 14 of the 16 totals


def _case(name, family, call, precision, stepping, packets, nx, ny, nz, optics=1.0, jobs=0, mix=0):
    c = {"family": family, "call": call, "precision": precision, "stepping": stepping, "packets": packets,
         "nx": nx, "ny": ny, "nz": nz, "optics": optics, "jobs": jobs, "mix": mix}
    return dict(c, name=name) if name else c


def listed():
    return [
        # an interactive preview: a small one-shot call, latency counts
        _case("sphere_preview_1e4", "sphere", "run", "mixed", W.SEGMENT, 10_000, 50, 50, 50),
        # one small block of a program that forbids device allocations, on a ragged grid
        _case("container_noalloc_1e4", "container", "noalloc", "mixed", W.SEGMENT, 10_000, 97, 50, 113),
        # plain FP64 with the paper's sphere tracing: the reference-accuracy run of a turbid sphere
        _case("sphere_fp64_1e5", "sphere", "run", "fp64", W.SPHERE_TRACING, 100_000, 50, 50, 50),
        # layered tissue in plain FP64 with per-packet records: a parity study
        _case("slab_fp64_1e5", "slab", "records", "fp64", W.SEGMENT, 100_000, 100, 100, 100),
        # a vessel network in plain FP64: many capsules under a smooth union
        _case("vessel_fp64_1e4", "vessel", "launch", "fp64", W.SEGMENT, 10_000, 100, 100, 100),
        # layered tissue at the size of the benchmark's step: the throughput case
        _case("slab_1e7", "slab", "launch", "mixed", W.SEGMENT, 10_000_000, 100, 100, 100),
        # the same tissue with the paper's own step rule
        _case("slab_tracing_1e6", "slab", "launch", "mixed", W.SPHERE_TRACING, 1_000_000, 100, 100, 100),
        # one launch of a vessel-network study (the full study is a series of such id blocks)
        _case("vessel_4e6", "vessel", "launch", "mixed", W.SEGMENT, 4_000_000, 200, 200, 200),
        # one launch of a curved glass container study: grazing incidence, clear shell
        _case("container_4e6", "container", "launch", "mixed", W.SEGMENT, 4_000_000, 128, 128, 128),
        # the shape gallery (tori, cylinders, frames, domain operations) end to end with a host grid
        _case("gallery_5e5", "gallery", "run", "mixed", W.SEGMENT, 500_000, 100, 100, 100),
        # the validation slab of the timing table: optically thick, 200 x 200 x 400 grid
        _case("jacques630_1e6", "jacques630", "launch", "mixed", W.SEGMENT, 1_000_000, 200, 200, 400),
        # a burst of jobs of all families served together
        _case("served_mix_10", "mix", "serve", "mixed", W.SEGMENT, 0, 0, 0, 0, jobs=10, mix=46),
    ]


# Per packet, with segment stepping / sphere tracing: steps, interactions,
# interfaces, voxel pieces (on a grid of `side` voxels across), and the
# arithmetic of one scene evaluation (box 20, sphere 8, capsule 22, bounding
# box 20, 5 per region; of a large union only the few nearest primitives).
EVENTS = {
    "sphere":     ((35, 29, 2.8, 137), (131, 29, 2.8, 220), 50, 33),
    "slab":       ((130, 115, 6.7, 257), (290, 115, 6.7, 360), 100, 95),
    "vessel":     ((108, 72, 3.9, 517), (210, 72, 3.9, 586), 200, 150),
    "container":  ((142, 130, 5.8, 382), (285, 130, 5.8, 515), 128, 54),
    "gallery":    ((146, 114, 4.3, 418), (251, 114, 4.3, 496), 100, 220),
    "jacques630": ((1458, 1452, 2.8, 582), (1498, 1452, 2.8, 587), 250, 45),
    "iso10":      ((60, 57, 1.0, 961), (101, 57, 1.0, 993), 200, 33),
    "beam":       ((5, 0, 2.0, 220), (41, 0, 2.0, 254), 200, 33),
}
# Most packets of a drawn case, mixed (segment stepping) and FP64.
MOST = {"sphere": (3e6, 6e4), "slab": (4e6, 6e4), "vessel": (1.5e6, 2e3), "container": (2e6, 4e4),
        "gallery": (3e5, 0), "jacques630": (4e5, 0), "iso10": (2e6, 6e4), "beam": (1e7, 6e5)}


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    stepping = rng.choice([W.SEGMENT, W.SEGMENT, W.SPHERE_TRACING])
    if rng.random() < 0.12:
        return _case("", "mix", "serve", "mixed", stepping, 0, 0, 0, 0, jobs=rng.randint(2, 6),
                     mix=rng.randint(5, 10_000))
    family = rng.choice(sorted(EVENTS))
    call = rng.choice(["launch", "launch", "records", "run", "run", "noalloc"])
    precision = "fp64" if MOST[family][1] > 0 and rng.random() < 0.35 else "mixed"
    most = MOST[family][precision == "fp64"] / (1 if stepping == W.SEGMENT else 2)
    n = between(500, most)
    nx, ny, nz = (between(16, 200) for _ in range(3))
    optics = round(rng.uniform(0.6, 1.2), 3)
    if call == "noalloc" and family == "vessel":   # 65 primitives: the fixed scratch holds them, the cell list not
        n = min(n, 200_000 if precision == "mixed" else 2_000)
    return _case("", family, call, precision, stepping, n, nx, ny, nz, optics)


def _workload(case, seed):
    """The case's workload with the packet stream of this seed."""
    n, fam = int(case["packets"]), case["family"]
    key = W.splitmix64(int(seed))
    wl = {"sphere": W.sphere_pencil, "slab": W.three_layer_slab, "vessel": W.vessel_network,
          "container": W.glass_container, "gallery": W.sdf_gallery,
          "jacques630": lambda: W.jacques_slab(630), "iso10": lambda: W.iso_sphere(10.0),
          "beam": W.glass_sphere_beam}[fam]()
    regions = tuple(replace(r, mu_s=r.mu_s * float(case["optics"])) for r in wl.scene.regions)
    g = wl.grid
    wl = replace(wl, npackets=n, seed=key, precision=case["precision"], scene=replace(wl.scene, regions=regions),
                 grid=W.Grid(g.lo, g.hi, (int(case["nx"]), int(case["ny"]), int(case["nz"]))))
    return wl.with_stepping(case["stepping"])


def _jobs(case, seed):
    """Jobs of the served mix with this seed's packet streams."""
    jobs = W.served_mix(int(case["jobs"]), int(case["mix"]), 1e4, 5e5, case["stepping"])
    return [replace(w, seed=W.splitmix64((int(seed) << 16) + j)) for j, w in enumerate(jobs)]


def prepare(case, seed):
    call = case["call"]
    if call == "serve":
        ctx = smc.Context(0)
        ctx.wait(ctx.submit(W.three_layer_slab(10_000).with_stepping(case["stepping"]), "mixed"))   # serving already
        return {"call": call, "ctx": ctx, "jobs": _jobs(case, seed)}
    wl = _workload(case, seed)
    s = {"call": call, "wl": wl}
    if call == "run":
        s["ctx"] = smc.Context(0)
        return s
    s["flu"] = torch.zeros(wl.grid.n[::-1], dtype=torch.int64, device="cuda")
    s["tot"] = smc.totals_tensor()
    if call != "noalloc":
        s["ctx"] = smc.Context(0)
        s["plan"] = s["ctx"].plan(wl, wl.precision)
        if call == "records":
            s["rec"] = torch.zeros((wl.npackets, 8), dtype=torch.int64, device="cuda")
    return s


def _counts(totals):
    return np.array([totals[f] for f in RESULTS], dtype=np.int64)


def run(state):
    call = state["call"]
    if call == "serve":
        ctx = state["ctx"]
        ids = [ctx.submit(w) for w in state["jobs"]]
        out = []
        for j in ids:
            fluence, totals, _latency = ctx.wait(j)
            out.append((fluence, _counts(totals)))
        return out
    wl = state["wl"]
    if call == "run":
        fluence, totals = state["ctx"].run(wl)
        return {"fluence": fluence, "totals": _counts(totals)}
    flu, tot = state["flu"], state["tot"]
    flu.zero_()
    tot.zero_()
    if call == "noalloc":
        smc.run_noalloc(wl, 0, wl.npackets, wl.seed, flu, tot)
    else:
        state["plan"].launch(0, wl.npackets, wl.seed, flu, tot, state.get("rec"))
    out = {"fluence": flu, "totals": tot[:NRESULTS]}
    if call == "records":
        out["records"] = state["rec"]
    return out


def _work(family, stepping, n, nx, ny, nz, optics):
    ev, tracing, side, per_eval = EVENTS[family]
    if stepping == W.SPHERE_TRACING:
        ev = tracing
    steps, scatters, interfaces, pieces = (e * (optics if k < 2 else 1.0) for k, e in enumerate(ev))
    pieces = pieces * (nx * ny * nz) ** (1 / 3) / side
    flops = steps * (48 + per_eval) + scatters * 62 + interfaces * (30 + 2 * per_eval) + pieces * 16
    return {"bytes": 8 * nx * ny * nz + 128, "flops": flops * n}


def work(case):
    if case["call"] == "serve":
        w = {"bytes": 0, "flops": 0}
        for j in _jobs(case, 0):
            fam = {1: "sphere", 2: "container", 3: "slab"}.get(len(j.scene.prims), "vessel")
            k = _work(fam, case["stepping"], j.npackets, *j.grid.n, 1.0)
            w = {q: w[q] + k[q] for q in w}
        return w
    w = _work(case["family"], case["stepping"], case["packets"], case["nx"], case["ny"], case["nz"], case["optics"])
    if case["call"] == "records":
        w["bytes"] += 64 * case["packets"]
    return w


def exact(case, seed):
    """Every output is a whole number that has to come out the same; none has a value in 64 bits to be compared with."""
    return None
