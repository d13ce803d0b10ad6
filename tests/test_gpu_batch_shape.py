"""Block sizes of mixed batches of many short series: blocks below four warps
only where there are no more of them than SMs, and the same results as the large
block bit for bit on the shapes that the model takes."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
RHO = synth.RHO_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("n,lo,hi", [(20, 100, 600), (1000, 100, 600), (4000, 300, 640), (6000, 10, 100)])
@pytest.mark.parametrize("rho", [0.0, RHO])
@pytest.mark.parametrize("n_md", [4, 50])
def test_small_blocks_only_one_to_an_SM(n, lo, hi, rho, n_md):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = np.random.default_rng(1).integers(lo, hi + 1, n)
    off = np.concatenate([[0], np.cumsum(T)])
    N = int(off[-1])
    th = synth.THETA_STD
    s = synth.rsv_series(N, th, seed=1)     # any values do: the series are cut from it
    y, lr = dev(s.y), dev(s.lnrv)
    rsv.rsv_set_leverage(ctx, rho)
    out = []
    for fixed in (False, True):
        if fixed:
            rsv.rsv_set_schedule(ctx, 384, 20, 384 * 20 - 2 * (n_md + 1) - 3)
        plan = rsv.Plan(ctx, off, n_md, prec="mixed")
        rsv.rsv_set_schedule(ctx)
        i = plan.info()
        if not fixed:
            assert i["threads"] >= 128 or i["bins"] <= sms, i
        h, dH = dev(s.h_true), torch.empty(2, n, dtype=torch.float64, device="cuda")
        acc = torch.empty(2, n, dtype=torch.int32, device="cuda")
        rsv.rsv_hmc_batched(ctx, plan, h, y, lr, dev([th] * n), 0.01, seed=3, n_traj=2, dH_out=dH, accept_out=acc)
        rsv.rsv_sync_status(ctx)
        out.append((h, dH, acc))
        plan.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    ctx.close()
