"""The FP64 path's fixed-point exponential at the edges of its range: the
switch to CUDA's exp at |t| = 128, arguments below its 2^-56 unit, the floors
of the reduction by ln2/1024, and the non-finite arguments.

Bound: the result is rounded once (0.5 ulp); the argument's truncation to
2^-56 (1/8 ulp of results below 1, half of that above), the reduction and the
table add less than 0.15 ulp, so it is within 0.65 ulp of e^t, and numpy's exp
is within 1 ulp: 1.65 ulp, and exactly 1 ulp apart at most where both round
to neighbours (2 ulp allows a numpy of 1 ulp error)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LN2 = np.log(2.0)
EDGES = {
    "switch": np.concatenate([np.nextafter(128.0, [0.0, 1e9]), [128.0], np.linspace(127.5, 128.5, 4001)]),
    "tiny": np.concatenate([2.0 ** -np.arange(40.0, 80.0), [5e-324, 1e-300, 0.0]]),
    "floors": np.concatenate([np.nextafter(np.arange(1, 6000) * (LN2 / 1024), d) for d in (0.0, 1e9)]),
    "octaves": np.concatenate([np.nextafter(np.arange(1, 184) * LN2, d) for d in (0.0, 1e9)]),
}


@pytest.mark.parametrize("name", list(EDGES))
def test_exponential_at_the_edges(name):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    t = np.concatenate([EDGES[name], -EDGES[name]])
    out = rsv.rsv_fp64_exp(ctx, torch.tensor(t, device="cuda")).cpu().numpy()
    ref = np.exp(t)
    assert np.max(np.abs(out - ref) / np.spacing(ref)) <= 2.0
    bad = rsv.rsv_fp64_exp(ctx, torch.tensor([np.inf, -np.inf, np.nan], dtype=torch.float64, device="cuda"))
    assert np.array_equal(bad.cpu().numpy(), [np.inf, 0.0, np.nan], equal_nan=True)
    ctx.close()
