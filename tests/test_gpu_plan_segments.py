"""Plans of many segments: thousands of series shorter than a warp's run, and
steps so many that a tile owns a few dozen sites.

Tolerances as everywhere: FP64 1e-12 relative on h' and 1e-9 on dH, mixed 1e-4
and 1e-3."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("prec,tol_h,tol_dh", [("fp64", 1e-12, 1e-9), ("mixed", 1e-4, 1e-3)])
def test_thousands_of_tiny_series(prec, tol_h, tol_dh):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    n, n_md, dtau, th = 5200, 6, 0.05, synth.THETA_STD
    T = np.random.default_rng(0).integers(1, 11, n)
    off = np.concatenate([[0], np.cumsum(T)])
    N = int(off[-1])
    assert n > N // 64 + 4096
    one = synth.rsv_series(N, th, seed=1)  # any values do: the series are cut from it
    p0 = synth.standard_normals(N, 2)
    rsv.rsv_reserve(ctx, N, n)
    plan = rsv.Plan(ctx, off, n_md, prec=prec)
    h, p = dev(one.h_true), dev(p0)
    dH = torch.empty(n, dtype=torch.float64, device="cuda")
    rsv.rsv_hmc_batched(ctx, plan, h, dev(one.y), dev(one.lnrv), dev([th] * n), dtau, p=p, log_u=dev([-1e300] * n), dH_out=dH)
    rsv.rsv_sync_status(ctx)
    h, dH = h.cpu().numpy(), dH.cpu().numpy()
    for s in range(n):
        a, b = off[s], off[s + 1]
        y, lr = one.y[a:b], one.lnrv[a:b]
        h1, p1 = oracle.leapfrog(one.h_true[a:b], p0[a:b], y, lr, th, n_md, dtau)
        assert np.max(np.abs(h[a:b] - h1) / np.maximum(1.0, np.abs(h1))) <= tol_h
        assert abs(dH[s] - oracle.delta_H(one.h_true[a:b], p0[a:b], h1, p1, y, lr, th)) <= tol_dh
    plan.close()
    ctx.close()


@pytest.mark.parametrize("prec,n_md,total", [("mixed", 3820, 330000), ("fp64", 3570, 160000)])
def test_tiles_of_a_few_sites_are_accepted(prec, n_md, total):
    """Windows that hold the series only in more tiles than the workspace is
    reserved for still make a plan, on the largest block."""
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    plan = rsv.Plan(ctx, [0, total - 100, total], n_md, prec=prec)
    i = plan.info()
    assert (i["threads"], i["sites_per_thread"]) == ((384, 20) if prec == "mixed" else (256, 28))
    assert i["split_series"] == 1 and i["bins"] > total // 64 + 4096
    plan.close()
    ctx.close()
