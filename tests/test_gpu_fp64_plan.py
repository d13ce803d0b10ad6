"""FP64 trajectories on the planner's short runs (one and two sites per thread)
and their neighbours, drawn momenta included, against the FP64 oracle.

Tolerances as everywhere for the FP64 path: 1e-12 relative on h' and 1e-9 on
dH for one trajectory; 1e-11 on h after a chain of three."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.fixture(scope="module")
def ctx():
    from paper_1603_08114_gb300 import rsv
    c = rsv.Context(0)
    yield c
    c.close()


# (T, n_md, sites per thread the planner takes): the smallest series, tiles of
# a few sites, an odd size, both sides of the step from one site to two
@pytest.mark.parametrize("T,n_md,j", [(1, 3, 1), (5, 1, 1), (129, 25, 1), (2000, 50, 1), (9001, 35, 1),
                                      (30001, 50, 2), (100003, 70, 4)])
@pytest.mark.parametrize("mass", [False, True])
def test_chain_with_drawn_momenta(ctx, T, n_md, j, mass):
    from paper_1603_08114_gb300 import rsv
    n, dtau = 3, 0.4 / n_md
    s = synth.rsv_series(T, TH, seed=T)
    minv = np.random.default_rng(2).uniform(0.5, 2.0, T).astype(np.float32) if mass else None
    assert rsv.rsv_chain_schedule(ctx, T, n_md, "fp64", with_mass=mass)["sites_per_thread"] == j
    h = dev(s.h_true)
    dH = torch.empty(n, dtype=torch.float64, device="cuda")
    rsv.rsv_hmc_chain(ctx, h, dev(s.y), dev(s.lnrv), dev(TH), n_md, dtau, n, prec="fp64", seed=5,
                      minv=dev(minv, torch.float32) if mass else None, dH_out=dH)
    rsv.rsv_sync_status(ctx)
    r = oracle.chain(s.h_true, s.y, s.lnrv, TH, n_md, dtau, 5, n, minv=None if minv is None else minv.astype(np.float64))
    assert np.max(np.abs(dH.cpu().numpy() - r["dH"])) <= 1e-9
    assert np.max(np.abs(h.cpu().numpy() - r["h"]) / np.maximum(1.0, np.abs(r["h"]))) < 1e-11


@pytest.mark.parametrize("T,j", [(700, 1), (30001, 2)])
def test_leverage_with_given_momenta(ctx, T, j):
    from paper_1603_08114_gb300 import rsv
    n_md, dtau, rho = 50, 0.01, -0.4
    s = synth.rsv_series_leverage(T, TH, rho, seed=T)
    p0 = synth.standard_normals(T, 3)
    h, p = dev(s.h_true), dev(p0)
    rsv.rsv_set_leverage(ctx, rho)
    try:
        assert rsv.rsv_chain_schedule(ctx, T, n_md, "fp64")["sites_per_thread"] == j
        dH, acc = rsv.rsv_hmc_trajectory(ctx, h, p, dev(s.y), dev(s.lnrv), TH, n_md, dtau, log_u=dev([-1e300]))
        rsv.rsv_sync_status(ctx)
    finally:
        rsv.rsv_set_leverage(ctx, 0.0)
    h1, p1 = oracle.leapfrog(s.h_true, p0, s.y, s.lnrv, TH + (rho,), n_md, dtau)
    dHr = oracle.delta_H(s.h_true, p0, h1, p1, s.y, s.lnrv, TH + (rho,))
    assert abs(dH.item() - dHr) <= 1e-9
    assert np.max(np.abs(h.cpu().numpy() - h1) / np.maximum(1.0, np.abs(h1))) <= 1e-12


@pytest.mark.parametrize("T", [2000, 30001])
def test_the_planned_shape_as_a_fixed_schedule(ctx, T):
    """The shape rsv_chain_schedule reports, fixed by rsv_set_schedule, gives
    the same trajectory bit for bit."""
    from paper_1603_08114_gb300 import rsv
    s = synth.rsv_series(T, TH, seed=1)
    cs = rsv.rsv_chain_schedule(ctx, T, 50, "fp64")
    outs = []
    for fixed in (False, True):
        if fixed:
            rsv.rsv_set_schedule(ctx, cs["threads"], cs["sites_per_thread"], cs["tile"])
        try:
            h = dev(s.h_true)
            dH, _ = rsv.rsv_hmc_trajectory(ctx, h, None, dev(s.y), dev(s.lnrv), TH, 50, 0.01, seed=2, log_u=dev([-1e300]))
        finally:
            rsv.rsv_set_schedule(ctx)
        outs.append((h, dH))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
