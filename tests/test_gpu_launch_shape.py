"""Launch shapes that a caller chooses are the ones that run.  The totals'
busy cycles (summed over the warps) over the launch's time tell how many warps
worked at a time."""
import pytest

import paper_2112_08035_gb300 as smc
import workloads as W

pytestmark = pytest.mark.gpu


def _warps(plan, wl):
    """Busy warp cycles per nanosecond of the launch: proportional to the warps."""
    import torch
    tot = smc.totals_tensor()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    plan.launch(0, wl.npackets, 3, None, tot)                    # first launch: loads the kernel
    torch.cuda.synchronize()
    tot.zero_()
    t0.record()
    plan.launch(0, wl.npackets, 3, None, tot)
    t1.record()
    torch.cuda.synchronize()
    assert plan.status() == 0
    return smc.totals_from_tensor(tot)["busy_cycles"] / (t0.elapsed_time(t1) * 1e6)


@pytest.mark.parametrize("threads", [32, 64, 128])
def test_blocks_zero_means_all_resident_blocks(threads):
    """One block per SM against blocks = 0 with the same threads: at least two
    blocks of up to 128 threads are resident on an SM, so the second runs about
    that many times the warps; midway is the limit."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = smc.Context(0)
    wl = W.three_layer_slab(60_000, precision="fp64").with_stepping(W.SEGMENT)
    plan = ctx.plan(wl, "fp64")
    plan.set_launch(sms, threads)
    one = _warps(plan, wl)
    plan.set_launch(0, threads)
    assert _warps(plan, wl) > 1.5 * one
    plan.close()
    ctx.close()


def test_a_small_trial_leaves_large_launches_their_shape():
    """FP64, 5000 packets: one block per SM is fastest (13.3 against 17.6 ms
    at 1e4), and the tuner reports it; a launch of 2^19 packets, of this plan
    or of a later one of the same shape, runs at least twice the warps."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ctx = smc.Context(0)
    small = W.three_layer_slab(5_000, precision="fp64").with_stepping(W.SEGMENT)
    large = small.with_packets(1 << 19)
    plan = ctx.plan(small, "fp64")
    blocks, threads, variant = plan.autotune(small.npackets)
    assert blocks == sms and threads in (64, 128) and variant in range(3)
    one = ctx.plan(large, "fp64")
    one.set_launch(sms, 128)
    few = _warps(one, large)
    for p in (plan, ctx.plan(large, "fp64")):
        assert _warps(p, large) > 1.5 * few
        p.close()
    one.close()
    ctx.close()
