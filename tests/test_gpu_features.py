"""Features and targets at the edges of their kernels -- series shorter than
the hbar window, blocks of 256 sites and their neighbours, a constant column --
against the FP64 reference, and the mass at the ends of a warp's 32 sites.

Tolerances: the reference standardises in FP64; the kernel rounds the raw
feature, its mean and 1/sd to FP32 (three roundings of 2^-24 on values of at
most 8, amplified by |mean|/sd <= 30 here): 2e-5, as in the existing test.  The
log scale is an FP32 rounding of an FP64 mean: 2^-24 of 4."""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("T", [1, 2, 3, 5, 31, 32, 33, 255, 256, 257, 513, 20011])
@pytest.mark.parametrize("flat", [False, True])
def test_features_and_mass(T, flat):
    from paper_1603_08114_gb300 import learned, rsv
    ctx = rsv.Context(0)
    s = synth.rsv_series(T, TH, seed=T)
    y = np.zeros(T) if flat else s.y     # y = 0: y^2 and its return term are constant columns
    F, st = rsv.rsv_mass_features(ctx, dev(y), dev(s.lnrv), dev(s.h_true), TH)
    ref, m, inv = mlp.standardize(mlp.features_raw(y, s.lnrv, s.h_true, s.theta))
    big = np.abs(inv) < 1e4              # a column of two nearly equal values has no bounded |mean|/sd
    assert np.max(np.abs(F.cpu().numpy() - ref)[:, big]) < 2e-5
    assert np.allclose(st.cpu().numpy()[:20], m, rtol=1e-6, atol=1e-6)
    P = learned.glorot_params(0)
    mo = torch.empty(T, dtype=torch.float32, device="cuda")
    minv = rsv.rsv_mlp_mass(ctx, F, dev(P, torch.float32), dev(y), dev(s.h_true), TH, m_out=mo,
                            log_scale=dev([3.4], torch.float32))
    lo, hi = mlp.mass_bounds(y, s.h_true, TH)
    mo, minv = mo.cpu().numpy(), minv.cpu().numpy()
    assert np.all(mo >= lo * (1 - 1e-6)) and np.all(mo <= hi * (1 + 1e-6))
    assert np.allclose(minv * mo, 1.0, rtol=1e-6)
    ctx.close()


@pytest.mark.parametrize("T", [1, 255, 256, 257, 400001])
def test_log_scale_is_the_mean_target(T):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    r = np.random.default_rng(T)
    m2 = r.uniform(1.0, 3.0, T)
    ls = torch.empty(1, dtype=torch.float32, device="cuda")
    hb = torch.empty(T, dtype=torch.float64, device="cuda")
    tgt = rsv.rsv_welford_target(ctx, dev(r.normal(size=T)), dev(m2), 100, hbar_out=hb, log_scale_out=ls)
    ref = np.log(99.0 / m2)
    assert np.max(np.abs(tgt.cpu().numpy() - ref)) <= 2.0 ** -24 * 5
    assert abs(ls.item() - tgt.cpu().numpy().astype(np.float64).mean()) <= 2.0 ** -24 * 5
    again = rsv.rsv_welford_target(ctx, dev(r.normal(size=T)), dev(m2), 100)
    assert torch.equal(again, tgt)
    ctx.close()
