"""A training whose device-side wait runs out never passes for a mass, and the
check that learned.train_mass makes for it keeps a non-finite dH of an earlier
call for the program's own rsv_sync_status."""
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
