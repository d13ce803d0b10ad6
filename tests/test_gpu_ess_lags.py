"""ESS where its passes end: fewer samples than a pass has lags, one more and
one fewer, series of odd lengths and few sites, slow columns that need many
passes, against the numpy estimator in FP64.

Tolerance as in the existing test: 1e-3 of the estimate for FP32 sums; a
truncation point may move by a pair on a few columns whose pair sum is near 0
(0.5 % of them, at least one)."""
import numpy as np
import pytest
import torch

from oracle import stats

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 7, 8, 9, 15, 16, 17, 63, 65, 300])
@pytest.mark.parametrize("T", [1, 31, 33, 9800, 40001])
def test_ess(n, T):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    r = np.random.default_rng(n * T)
    rho = r.uniform(-0.3, 0.98, T)
    x = np.empty((n, T))
    x[0] = r.standard_normal(T) / np.sqrt(1 - rho ** 2)
    for k in range(1, n):
        x[k] = rho * x[k - 1] + r.standard_normal(T)
    if T > 5:
        x[:, 5] = 1.25
    x = x.astype(np.float32)
    got = rsv.rsv_ess(ctx, torch.tensor(x, device="cuda")).cpu().numpy()
    ref = stats.ess_geyer(x.astype(np.float64))
    far = np.abs(got - ref) > 1e-3 * np.maximum(ref, 1.0)
    assert far.sum() <= max(1, 0.005 * T) and np.median(np.abs(got - ref) / np.maximum(ref, 1.0)) < 1e-5
    ctx.close()
