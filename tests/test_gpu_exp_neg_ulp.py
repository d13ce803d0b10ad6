"""exp_neg's stated bound, 0.65 ulp, against e^t to 40 digits: arguments over the
range of the integer form, near 0 (where the truncation of the argument weighs
most), just below powers of two of the result, and at the form's own limit."""
import math
from decimal import Decimal, localcontext

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_within_the_stated_bound():
    from paper_1603_08114_gb300 import rsv
    r = np.random.default_rng(0)
    ln2 = math.log(2.0)
    t = np.concatenate([r.uniform(-128, 128, 12000), r.normal(0, 3, 6000), -np.exp(r.uniform(-45, 0, 4000)),
                        r.integers(-180, 180, 3000) * ln2 - np.exp(r.uniform(-38, -4, 3000)),
                        [-127.99999999999999, 127.99999999999999, -0.0, 0.0, -2.0 ** -60, 2.0 ** -60]])
    ctx = rsv.Context(0)
    out = rsv.rsv_fp64_exp(ctx, torch.tensor(t, dtype=torch.float64, device="cuda")).cpu().numpy()
    worst = 0.0
    with localcontext() as c:
        c.prec = 40
        for a, b in zip(t.tolist(), out.tolist()):
            e = Decimal(a).exp()
            worst = max(worst, float(abs(Decimal(b) - e) / Decimal(math.ulp(float(e)))))
    assert worst <= 0.65, worst
    ctx.close()
