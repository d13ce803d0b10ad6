"""rsv_reserve(max_T, max_series) covers every smaller call: under stream
capture, where a workspace that had to grow is refused, such calls are
recorded, and the replay gives what the call itself gives, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def captured(call):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    g.replay()
    torch.cuda.synchronize()


# both sides of 152 x 256 sites, where a block of the sweep takes four times as many
@pytest.mark.parametrize("max_T", [38912, 38913, 40000, 100000, 155000, 160000])
@pytest.mark.parametrize("T", [2000, 25089, 38912, 38913])
def test_theta_sweep_of_fewer_sites(max_T, T):
    from paper_1603_08114_gb300 import rsv
    if T > max_T:
        pytest.skip("longer than the reserve")
    s = synth.rsv_series(T, TH, seed=3)
    h, lr, th0 = dev(s.h_true), dev(s.lnrv), dev(TH)
    plain, fresh = rsv.Context(0), rsv.Context(0)
    ref = th0.clone()
    rsv.rsv_gibbs_theta(plain, h, lr, ref, seed=5, traj=2)
    rsv.rsv_reserve(fresh, max_T, 1)
    th = th0.clone()
    captured(lambda: rsv.rsv_gibbs_theta(fresh, h, lr, th, seed=5, traj=2))
    assert torch.equal(th, ref)
    plain.close()
    fresh.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_thousands_of_tiny_series(prec):
    from paper_1603_08114_gb300 import rsv
    n = 5200
    off = np.concatenate([[0], np.cumsum(np.random.default_rng(0).integers(1, 11, n))])
    N = int(off[-1])
    s = synth.rsv_series(N, TH, seed=1)
    y, lr, th = dev(s.y), dev(s.lnrv), dev([TH] * n)
    out = []
    for capture in (False, True):
        ctx = rsv.Context(0)
        rsv.rsv_reserve(ctx, N, n)
        plan = rsv.Plan(ctx, off, 6, prec=prec)
        h, acc = dev(s.h_true), torch.empty(n, dtype=torch.int32, device="cuda")

        def call():
            rsv.rsv_hmc_batched(ctx, plan, h, y, lr, th, 0.05, seed=4, accept_out=acc)
        captured(call) if capture else call()
        torch.cuda.synchronize()
        out.append((h, acc))
        plan.close()
        ctx.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
