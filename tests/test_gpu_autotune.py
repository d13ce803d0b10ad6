"""A tuned plan is never slower than the planner's own, which is measured first
(up to the spread of two measurements of a plan, far below the several times
that the shapes differ by here), and a cached choice makes the same plan."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def time_us(rsv, ctx, plan, h0, y, lr, th):
    ts = []
    for r in range(8):
        h = h0.clone()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        rsv.rsv_hmc_batched(ctx, plan, h, y, lr, th, 0.02, seed=1, traj0=r)
        b.record()
        b.synchronize()
        ts.append(1e3 * a.elapsed_time(b))
    return min(ts[2:])


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,lo,hi", [(64, 300, 2000), (10, 300, 1000)])
def test_tuned_plan_against_the_automatic_one(prec, n, lo, hi, tmp_path, monkeypatch):
    from paper_1603_08114_gb300 import autotune, rsv
    monkeypatch.setenv("RSV_TUNE_CACHE", str(tmp_path))
    ctx = rsv.Context(0)
    b = synth.rsv_batch(n, lo, hi, seed=2)
    y, lr, th, h0 = dev(b.y), dev(b.lnrv), dev(b.theta.ravel()), dev(b.h_true)
    args = (ctx, b.offsets, 50, prec, y, lr, th, 0.02, h0)
    plan, sched = autotune.tune_plan(*args)
    auto = rsv.Plan(ctx, b.offsets, 50, prec)
    assert time_us(rsv, ctx, plan, h0, y, lr, th) <= 1.25 * time_us(rsv, ctx, auto, h0, y, lr, th)
    i = auto.info()
    assert any(c[1:] == (i["threads"], i["sites_per_thread"], True) for c in sched["candidates"])
    again, cached = autotune.tune_plan(*args)
    assert cached["cached"] and again.info() == plan.info()
    assert (cached["threads"], cached["sites_per_thread"]) == (sched["threads"], sched["sites_per_thread"])
    for p in (plan, auto, again):
        p.close()
    ctx.close()


def test_integrators_whose_halo_no_fixed_shape_allows(tmp_path, monkeypatch):
    """Candidates that do not fit are left out; the automatic plan is always there."""
    from paper_1603_08114_gb300 import autotune, rsv
    monkeypatch.setenv("RSV_TUNE_CACHE", str(tmp_path))
    ctx = rsv.Context(0)
    rsv.rsv_set_integrator(ctx, "omelyan4")
    b = synth.rsv_batch(5, 200, 400, seed=3)
    plan, sched = autotune.tune_plan(ctx, b.offsets, 30, "fp64", dev(b.y), dev(b.lnrv), dev(b.theta.ravel()), 0.02, dev(b.h_true))
    assert sched["automatic"] and len(sched["candidates"]) >= 1
    plan.close()
    ctx.close()
