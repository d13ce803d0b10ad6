"""The states of a batch written back in parts of its segments: few segments of
many sites, ragged parts, segments shorter than the parts, accepted and rejected
series side by side -- the same bits as on tiles of another size, and a rejected
series untouched."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("prec,other", [("fp64", (64, 4)), ("mixed", (64, 8))])
@pytest.mark.parametrize("T", [[20011, 3], [7677, 1, 1025, 1024, 1023], [1, 2], [40000, 9, 15355], [300] * 700])
def test_parts_of_segments(prec, other, T):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    n, n_md, th = len(T), 5, synth.THETA_STD
    off = np.concatenate([[0], np.cumsum(T)])
    s = synth.rsv_series(int(off[-1]), th, seed=2)   # any values do: the series are cut from it
    p0 = synth.standard_normals(int(off[-1]), 3)
    lu = np.where(np.arange(n) % 3 == 1, 1e300, -1e300)   # every third series rejected
    out = []
    for shape in (None, other):
        if shape:
            rsv.rsv_set_schedule(ctx, shape[0], shape[1], shape[0] * shape[1] - 2 * (n_md + 1) - 3)
        plan = rsv.Plan(ctx, off, n_md, prec=prec)
        rsv.rsv_set_schedule(ctx)
        h, p = dev(s.h_true), dev(p0)
        rsv.rsv_hmc_batched(ctx, plan, h, dev(s.y), dev(s.lnrv), dev([th] * n), 0.02, p=p, log_u=dev(lu))
        rsv.rsv_sync_status(ctx)
        out.append(h)
        plan.close()
    assert torch.equal(out[0], out[1])
    h0 = dev(s.h_true)
    for i in range(n):
        same = torch.equal(out[0][off[i]:off[i + 1]], h0[off[i]:off[i + 1]])
        assert same == (i % 3 == 1), i
    ctx.close()
