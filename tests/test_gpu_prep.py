"""The mixed path's conversions at the boundary, on the integer units: a call of
no trajectories takes h to its (hi, lo) FP32 pair and back.  They round to
nearest even like the FP64 conversions, so the result is numpy's bit for bit:
halfway cases, carries into the exponent, signed zeros, subnormal and tiny
values (which the kernels hand to the conversions), large ones; and packed
series whose borders fall anywhere in the write-back's runs of 1024 sites."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
TH = (0.95, -0.5, -0.2, 0.05, 0.1)


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def edges(T):
    r = np.random.default_rng(T)
    f = r.normal(0, 2, T).astype(np.float32)
    half = np.spacing(f).astype(np.float64) / 2
    pool = np.concatenate([
        f.astype(np.float64), f + half, f - half, f + half * (1 + 2.0 ** -20), f + half * r.uniform(-1, 1, T),
        np.nextafter(2.0 ** np.arange(-30.0, 30), 0), -np.nextafter(2.0 ** np.arange(-30.0, 30), 0),
        [0.0, -0.0, 1e-30, -2.0 ** -73, 2.0 ** -74, 1e-45, 5e-324, 1e30, -1.5e38],
        r.normal(0, 1, T) * 2.0 ** r.integers(-90, 60, T)])
    r.shuffle(pool)
    return pool[:T]


@pytest.mark.parametrize("T", [1, 31, 1023, 1025, 5000, 70001])
@pytest.mark.parametrize("rho", [0.0, -0.4])
def test_state_goes_to_pairs_and_back(T, rho):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    h0 = edges(T)
    h = dev(h0)
    rsv.rsv_set_leverage(ctx, rho)
    rsv.rsv_hmc_chain(ctx, h, dev(np.zeros(T)), dev(edges(T)), dev(TH), 10, 0.01, 0, prec="mixed")
    torch.cuda.synchronize()
    hi = h0.astype(np.float32)
    lo = (h0 - hi.astype(np.float64)).astype(np.float32)
    assert np.array_equal(h.cpu().numpy(), hi.astype(np.float64) + lo.astype(np.float64))
    ctx.close()


def test_packed_series_go_back_to_their_places():
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    T = np.array([1, 2, 1021, 1024, 3, 1, 1, 2047, 9000, 5, 500])
    off = np.concatenate([[0], np.cumsum(T)])
    h0 = np.random.default_rng(0).normal(-0.5, 0.3, off[-1])
    h = dev(h0)
    plan = rsv.Plan(ctx, off, 10)
    rsv.rsv_hmc_batched(ctx, plan, h, dev(np.ones(off[-1])), dev(h0), dev([list(TH)] * len(T)), 0.01, n_traj=0)
    torch.cuda.synchronize()
    hi = h0.astype(np.float32)
    assert np.array_equal(h.cpu().numpy(), hi.astype(np.float64) + (h0 - hi).astype(np.float32))
    plan.close()
    ctx.close()
