"""rsv_welford_target keeps its block sums where nothing else of the context
writes or reallocates them: a captured call still gives the log scale after the
workspace has grown, and a chain on another stream is the same with target
calls beside it, bit for bit."""
import numpy as np
import torch
import pytest

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def moments(T):
    r = np.random.default_rng(T)
    return dev(r.normal(size=T)), dev(r.uniform(1.0, 3.0, T))


def test_captured_call_outlives_growth_of_the_workspace():
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    mean, m2 = moments(300001)
    ref, ls = torch.empty(1, device="cuda"), torch.empty(1, device="cuda")
    rsv.rsv_welford_target(ctx, mean, m2, 100, log_scale_out=ref)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rsv.rsv_welford_target(ctx, mean, m2, 100, log_scale_out=ls)
    rsv.rsv_reserve(ctx, 1 << 22, 100000)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(ls, ref)
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_chain_beside_target_calls(prec):
    from paper_1603_08114_gb300 import rsv
    T, n = 30001, 30
    s = synth.rsv_series(T, TH, seed=1)
    y, lr = dev(s.y), dev(s.lnrv)
    mean, m2 = moments(300001)
    side = torch.cuda.Stream()
    out = []
    for beside in (False, True):
        ctx = rsv.Context(0)
        h, th, ls = dev(s.h_true), dev(TH), torch.empty(1, device="cuda")
        dH = torch.empty(n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        if prec == "mixed":
            rsv.rsv_set_persistent(ctx, False)  # many launches for the other stream's to fall between
        rsv.rsv_hmc_chain(ctx, h, y, lr, th, 20, 0.02, n, prec=prec, seed=2, update_theta=True, dH_out=dH)
        with torch.cuda.stream(side):
            for _ in range(40 if beside else 1):
                rsv.rsv_welford_target(ctx, mean, m2, 100, log_scale_out=ls)
        torch.cuda.synchronize()
        out.append((h, th, dH, ls))
        ctx.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
