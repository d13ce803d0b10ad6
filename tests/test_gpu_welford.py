"""The per-site moments against the recurrence in numpy's FP64, row by row: the
kernel's division by the row count is the correctly rounded one, so mean and M2
agree bit for bit where the recurrence's last step is fused as the kernel's
is, and to a rounding of M2 otherwise: the mean exactly, M2 to n ulp.

Rows that are constant, zero or subnormal, far out, huge and tiny; one row,
more rows than a block holds counts for; appended rows."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rows(name, n, T):
    r = np.random.default_rng(n)
    x = -0.5 + 0.2 * r.standard_normal((n, T))
    x = {"plain": x, "near zero": 0.01 * x + 1e-3, "constant": np.full((n, T), 1.25), "zeros": 0.0 * x,
         "huge": 1e25 * (1 + x), "tiny": 1e-20 * x, "subnormal": 1e-42 * x, "offset": 1e6 + x}[name]
    return x.astype(np.float32)


@pytest.mark.parametrize("name", ["plain", "near zero", "constant", "zeros", "huge", "tiny", "subnormal", "offset"])
@pytest.mark.parametrize("n,split,T", [(1, 0, 1), (2, 0, 33), (8, 0, 257), (41, 13, 300), (600, 0, 65)])
def test_moments_are_the_recurrence(name, n, split, T):
    from paper_1603_08114_gb300 import rsv
    X = rows(name, n, T)
    ctx = rsv.Context(0)
    mean = torch.zeros(T, dtype=torch.float64, device="cuda")
    m2 = torch.zeros_like(mean)
    c = 0
    for part in ([X] if not split else [X[:split], X[split:]]):
        c = rsv.rsv_welford_update(ctx, torch.tensor(part, device="cuda"), c, mean, m2)
    ctx.close()
    assert c == n
    m, s = np.zeros(T), np.zeros(T)
    for k in range(n):
        v = X[k].astype(np.float64)
        d = v - m
        m = m + d / (k + 1)
        s = s + d * (v - m)
    assert np.array_equal(mean.cpu().numpy(), m)
    assert np.all(np.abs(m2.cpu().numpy() - s) <= n * np.spacing(s))
