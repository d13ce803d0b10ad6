"""ESS on both sides of the number of samples from which the lags are taken
several a pass, against an FP32 restatement of the arithmetic that both kernels
share -- compensated sums in sample order -- to 2 ulp (the divisions and the
logarithm)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
F = np.float32


def fma(a, b, c):
    """FP32 fused multiply-add: the product exact in FP64, the sum rounded there and to FP32."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def ess32(x):
    n, T = x.shape
    s, c = np.zeros(T, F), np.zeros(T, F)
    for k in range(n):
        v = x[k] - c
        q = s + v
        c = (q - s) - v
        s = q
    m = s / F(n)
    d = x - m

    def gamma(lag):
        a, ca = np.zeros(T, F), np.zeros(T, F)
        for k in range(n - lag):
            v = fma(d[k], d[k + lag], -ca)
            q = a + v
            ca = (q - a) - v
            a = q
        return a / F(n)
    g0 = gamma(0)
    go, prev, tau = g0 > 0, np.full(T, np.inf, F), np.zeros(T, F)
    with np.errstate(all="ignore"):
        for mm in range((n - 1 + 1) // 2):
            if 2 * mm + 1 >= n:
                break
            G = (F(1) if mm == 0 else gamma(2 * mm) / g0) + gamma(2 * mm + 1) / g0
            go &= G > 0
            prev = np.where(go, np.minimum(G, prev), prev)
            tau = np.where(go, tau + prev, tau).astype(F)
        t = np.maximum(F(-1) + F(2) * tau, F(1) / np.log10(F(max(n, 10))))
        return np.where(g0 > 0, F(n) / t, F(0))


@pytest.mark.parametrize("n", [2, 3, 4, 9, 11, 12, 13, 14])
@pytest.mark.parametrize("T", [1, 255, 257, 60001])
def test_both_sides_of_the_rule(n, T):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    r = np.random.default_rng(100 * n + T)
    x = np.cumsum(r.standard_normal((n, T)), axis=0) if n % 2 else r.standard_normal((n, T))
    x = x.astype(F)
    x[:, T // 2] = 0.75   # a column that never moves
    got = rsv.rsv_ess(ctx, torch.tensor(x, device="cuda")).cpu().numpy()
    ref = ess32(x)
    assert got[T // 2] == 0.0
    close = np.abs(got - ref) <= 2 * np.spacing(np.maximum(got, ref))
    # (an FMA restated in FP64 may round twice, and a pair sum near 0 then ends one pair earlier)
    assert close.mean() >= (1.0 if T < 1000 else 0.999)
    ctx.close()
