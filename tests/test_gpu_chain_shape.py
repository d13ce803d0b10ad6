"""Short series with few force evaluations: the chain's blocks have the warps that
its serial phases (draws, sweep, decision) need, and the chain on that shape is
the one of the series in a single block: states and theta bit for bit, dH to the
rounding of its sums (a few thousand terms of order 1 in double-float: 1e-9)."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("T", [200, 500, 1000, 2000, 2742])
@pytest.mark.parametrize("n_md,integrator", [(1, "leapfrog"), (3, "omelyan2"), (12, "leapfrog"), (25, "leapfrog")])
@pytest.mark.parametrize("mass", [False, True])
def test_blocks_of_several_warps(T, n_md, integrator, mass):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    rsv.rsv_set_integrator(ctx, integrator)
    cs = rsv.rsv_chain_schedule(ctx, T, n_md, "mixed", with_mass=mass)
    assert cs["persistent"] and cs["sites_per_thread"] == 4
    assert cs["threads"] >= min(96, 32 * -(-T // 128))
    s = synth.rsv_series(T, TH, seed=T)
    minv = dev(np.random.default_rng(1).uniform(0.5, 2.0, T), torch.float32) if mass else None
    n, out = 12, []
    for one in (False, True):
        if one:
            rsv.rsv_set_schedule(ctx, 32 * -(-T // 128), 4, T)
        h, th = dev(s.h_true), dev(TH)
        dH = torch.empty(n, dtype=torch.float64, device="cuda")
        rsv.rsv_hmc_chain(ctx, h, dev(s.y), dev(s.lnrv), th, n_md, 0.05, n, prec="mixed", minv=minv, seed=2, update_theta=True, dH_out=dH)
        rsv.rsv_sync_status(ctx)
        out.append((h, th, dH))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert (out[0][2] - out[1][2]).abs().max().item() <= 1e-9
    ctx.close()
