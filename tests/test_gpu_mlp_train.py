"""Training in one launch against the same Adam steps one call at a time (a call
of one step takes the step kernel): the arithmetic and the order of the sums
are the same, so the parameters agree to FP32 rounding of a step of lr
(1e-3 x 2^-23 a step, 1e-6 allows for hundreds).  Batches at the edges: one
block, fewer parameters than lanes per block, more partials than are staged
at a time, more blocks than can be resident."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH = synth.THETA_STD


@pytest.mark.parametrize("T,batch", [(1, 64), (777, 64), (5003, 192), (5003, 4096), (20000, 64 * 130), (20000, 64 * 1300)])
def test_training_in_one_launch_equals_single_steps(T, batch):
    from paper_1603_08114_gb300 import learned, rsv
    ctx = rsv.Context(0)
    rng = np.random.default_rng(T)
    feat = torch.tensor(rng.normal(size=(T, 20)).clip(-8, 8), dtype=torch.float32, device="cuda")
    target = torch.tensor(3.4 + 0.1 * rng.normal(size=T), dtype=torch.float32, device="cuda")
    ls = torch.tensor([3.4], dtype=torch.float32, device="cuda")
    n, out = 7, []
    for one in (True, False):
        P = torch.tensor(learned.glorot_params(1), device="cuda")
        m, v, loss = torch.zeros_like(P), torch.zeros_like(P), torch.full((n,), -1.0, device="cuda")
        if one:
            rsv.rsv_mlp_train(ctx, feat, target, P, m, v, 3, n, batch, 9, loss_out=loss, log_scale=ls)
        else:
            for i in range(n):
                rsv.rsv_mlp_train(ctx, feat, target, P, m, v, 3 + i, 1, batch, 9, loss_out=loss[i:], log_scale=ls)
        rsv.rsv_sync_status(ctx)
        out.append((P, m, v, loss))
    for a, b in zip(*out):
        assert torch.isfinite(a).all() and (a - b).abs().max().item() <= 1e-6 * max(1.0, b.abs().max().item())
    ctx.close()


def test_a_wait_that_runs_out_is_reported():
    from paper_1603_08114_gb300 import learned, rsv
    ctx = rsv.Context(0)
    feat, target = torch.zeros(500, 20, device="cuda"), torch.zeros(500, device="cuda")
    P = torch.tensor(learned.glorot_params(1), device="cuda")
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    rsv.rsv_set_wait_limit(ctx, 1)
    rsv.rsv_mlp_train(ctx, feat, target, P, m, v, 0, 50, 4096, 9)
    with pytest.raises(rsv.RSVError, match="RSV_ETIMEOUT"):
        rsv.rsv_sync_status(ctx)
    rsv.rsv_set_wait_limit(ctx, 0)
    rsv.rsv_mlp_train(ctx, feat, target, P, m, v, 0, 5, 4096, 9)
    rsv.rsv_sync_status(ctx)
    ctx.close()
