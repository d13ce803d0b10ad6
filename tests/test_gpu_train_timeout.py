"""A training whose device-side wait runs out never passes for a mass: train_mass
raises where the program has set a limit, and the mass is NaN until the timeout
is reported in any case.  The check keeps a non-finite dH of an earlier call for
the program's own rsv_sync_status."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.fixture
def setup():
    from paper_1603_08114_gb300 import learned, rsv
    ctx = rsv.Context(0)
    s = synth.rsv_series(3000, TH, seed=1)
    y, lr = dev(s.y), dev(s.lnrv)
    m2 = torch.full_like(y, 3.3)

    def train():
        return learned.train_mass(ctx, y, lr, TH, dev(s.h_true), m2, 100, steps=40, batch=4096)
    yield rsv, ctx, s, train
    ctx.close()


def test_a_wait_that_runs_out_is_raised(setup):
    rsv, ctx, s, train = setup
    good = train()
    rsv.rsv_set_wait_limit(ctx, 1)
    with pytest.raises(rsv.RSVError, match="RSV_ETIMEOUT"):
        train()
    rsv.rsv_set_wait_limit(ctx, 0)
    again = train()
    rsv.rsv_sync_status(ctx)
    assert torch.equal(again.minv, good.minv) and torch.equal(again.losses, good.losses)


def test_a_nonfinite_dH_is_still_reported(setup):
    rsv, ctx, s, train = setup
    y = s.y.copy()
    y[5] = np.inf
    rsv.rsv_set_wait_limit(ctx, 1 << 31)   # the default, set: train_mass checks
    for _ in range(2):
        rsv.rsv_hmc_trajectory(ctx, dev(s.h_true), None, dev(y), dev(s.lnrv), TH, 3, 0.02)
        train()
        with pytest.raises(rsv.RSVError, match="RSV_ENONFINITE"):
            rsv.rsv_sync_status(ctx)
        rsv.rsv_sync_status(ctx)
    rsv.rsv_hmc_trajectory(ctx, dev(s.h_true), None, dev(y), dev(s.lnrv), TH, 3, 0.02)
    train()
    assert rsv.rsv_sync_status(ctx, allow_nonfinite=True) == rsv.RSV_ENONFINITE
    assert rsv.rsv_sync_status(ctx) == rsv.RSV_OK


def test_the_mass_is_nan_until_the_timeout_is_reported(setup):
    from paper_1603_08114_gb300 import learned
    rsv, ctx, s, train = setup
    good = train()
    y, hb, ls = dev(s.y), dev(s.h_true), good.log_scale
    P = torch.tensor(learned.glorot_params(0), device="cuda")
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    mo = torch.empty(3000, dtype=torch.float32, device="cuda")
    rsv.rsv_set_wait_limit(ctx, 1)
    rsv.rsv_mlp_train(ctx, good.features, good.target, P, m, v, 0, 40, 4096, 0, log_scale=ls)
    rsv.rsv_set_wait_limit(ctx, 0)
    minv = rsv.rsv_mlp_mass(ctx, good.features, good.params, y, hb, TH, m_out=mo, log_scale=ls)
    assert torch.isnan(minv).all() and torch.isnan(mo).all()
    with pytest.raises(rsv.RSVError, match="RSV_ETIMEOUT"):
        rsv.rsv_sync_status(ctx)
    assert torch.equal(rsv.rsv_mlp_mass(ctx, good.features, good.params, y, hb, TH, log_scale=ls), good.minv)
