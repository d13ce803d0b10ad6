"""Statistics of the mass features where a one-pass variance would lose its
digits: a site far out at the middle or at an end (which some hbar columns
leave out), columns of zeros (series no longer than the hbar window), values
that differ little from a large mean.

Reference: numpy's two passes over the FP32 features.  Tolerance: the FP32
rounding of the result, 2^-24, and of one feature value that rounds the other
way (the kernel's exponential is within an ulp of FP64), 2^-24 of it: 2^-22.
FP64 sums add less than 1e-12 of a column's largest value to the mean."""
import numpy as np
import pytest
import torch

from oracle import mlp
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("T", [1, 2, 3, 4, 5, 7, 8, 9, 10, 12, 20, 255, 256, 257, 1000, 300001])
@pytest.mark.parametrize("kind", ["plain", "middle", "ends", "narrow"])
def test_statistics_match_two_passes(T, kind):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    s = synth.rsv_series(T, TH, seed=T)
    y, lr, hb = s.y.copy(), s.lnrv.copy(), s.h_true.copy()
    if kind == "middle":
        y[T // 2], lr[T // 2], hb[T // 2] = 2e4, -3e7, 1e6
    elif kind == "ends":
        hb[0] = 1e6
        hb[-1] = 3e5
        lr[0], y[-1] = 5e6, 1e4
    elif kind == "narrow":
        hb = 300.0 + 1e-3 * hb
        lr = -4e3 + 1e-2 * lr
    F, st = rsv.rsv_mass_features(ctx, dev(y), dev(lr), dev(hb), TH)
    raw = mlp.features_raw(y, lr, hb, TH).astype(np.float32).astype(np.float64)
    ref, m, inv = mlp.standardize(raw)
    st, tol = st.cpu().numpy().astype(np.float64), 2.0 ** -22
    assert np.all(np.abs(st[:20] - m) <= tol * np.abs(m) + 1e-12 * np.abs(raw).max(axis=0))
    assert np.all(np.abs(st[20:] - inv) <= tol * inv), (st[20:], inv)
    assert torch.isfinite(F).all()
    ctx.close()
