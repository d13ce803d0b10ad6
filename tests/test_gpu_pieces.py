"""S(h), dS/dh and the FP64 theta sweep where their kernels change shape: one
site per thread up to 38912 sites and runs of four beyond, a remainder of
every length, the smallest series; with and without leverage; states past the
exponential's range.

Tolerances as for these entry points elsewhere: 1e-13 of max(1, |F|) (1e-12
with leverage), 1e-12 of max(1, |S|), 1e-11 relative for a sweep's theta."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD
SIZES = [1, 2, 3, 4, 5, 63, 64, 65, 257, 2000, 38911, 38912, 38913, 38914, 38915, 38916, 100003]


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.fixture(scope="module")
def ctx():
    from paper_1603_08114_gb300 import rsv
    c = rsv.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("T", SIZES)
@pytest.mark.parametrize("rho", [0.0, -0.4])
def test_force_and_action(ctx, T, rho):
    from paper_1603_08114_gb300 import rsv
    s = synth.rsv_series_leverage(T, TH, rho, seed=T) if rho else synth.rsv_series(T, TH, seed=T)
    h = s.h_true + 0.2 * synth.standard_normals(T, 3)
    th = TH + (rho,) if rho else TH
    rsv.rsv_set_leverage(ctx, rho)
    try:
        F = rsv.rsv_force(ctx, dev(h), dev(s.y), dev(s.lnrv), TH).cpu().numpy()
        S = rsv.rsv_action(ctx, dev(h), dev(s.y), dev(s.lnrv), TH).item()
    finally:
        rsv.rsv_set_leverage(ctx, 0.0)
    ref = oracle.force(h, s.y, s.lnrv, th)
    assert np.max(np.abs(F - ref) / np.maximum(1.0, np.abs(ref))) < (1e-12 if rho else 1e-13)
    r = oracle.action(h, s.y, s.lnrv, th)
    assert abs(S - r) <= 1e-12 * max(1.0, abs(r))


@pytest.mark.parametrize("T", [5, 40000])
def test_states_past_the_range_of_the_exponential(ctx, T):
    from paper_1603_08114_gb300 import rsv
    s = synth.rsv_series(T, TH, seed=T)
    h = s.h_true.copy()
    h[:5] = [300.0, -200.0, 128.0, -128.0, 0.0]
    F = rsv.rsv_force(ctx, dev(h), dev(s.y), dev(s.lnrv), TH).cpu().numpy()
    ref = oracle.force(h, s.y, s.lnrv, TH)
    assert np.max(np.abs(F - ref) / np.maximum(1.0, np.abs(ref))) < 1e-12
    S, r = rsv.rsv_action(ctx, dev(h), dev(s.y), dev(s.lnrv), TH).item(), oracle.action(h, s.y, s.lnrv, TH)
    assert abs(S - r) <= 1e-12 * abs(r)


@pytest.mark.parametrize("T", SIZES)
def test_theta_sweep(ctx, T):
    from paper_1603_08114_gb300 import rsv
    s = synth.rsv_series(T, TH, seed=T + 7)
    th = dev(TH)
    for k in range(2):  # the second sweep reuses the counter and the scratch
        before = th.cpu().numpy()
        rsv.rsv_gibbs_theta(ctx, dev(s.h_true), dev(s.lnrv), th, seed=3, traj=k)
        ref, _ = oracle.gibbs_theta(s.h_true, s.lnrv, before, 3, 0, k)
        assert np.max(np.abs(th.cpu().numpy() - ref) / np.maximum(1e-3, np.abs(ref))) < 1e-11
