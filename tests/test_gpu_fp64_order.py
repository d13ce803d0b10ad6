"""An FP64 series' results are the same bits whatever it is packed with and
whatever block shape or tiles it lands on: dH is summed free of order.  And
terms too large for that sum, where an energy is far outside its usual range,
against the oracle: 1e-12 of the largest term."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
SHAPES = [None, (32, 1), (128, 1), (64, 2), (192, 2), (96, 4), (256, 4), (64, 8), (160, 16), (128, 28), (256, 28)]


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def batched(rsv, ctx, T, ths, ser, n_md, shape, rows, minv=None):
    """(h, dH, accept) of the packed series, three trajectories with drawn momenta."""
    off = np.concatenate([[0], np.cumsum(T)])
    if shape is not None:
        rsv.rsv_set_schedule(ctx, shape[0], shape[1], shape[0] * shape[1] - 2 * (n_md + 1) - 3)
    try:
        plan = rsv.Plan(ctx, off, n_md, prec="fp64", with_mass=minv is not None)
    finally:
        rsv.rsv_set_schedule(ctx)
    h, dH = dev(np.concatenate([s.h_true for s in ser])), torch.empty(rows, len(T), dtype=torch.float64, device="cuda")
    acc = torch.empty(rows, len(T), dtype=torch.int32, device="cuda")
    rsv.rsv_hmc_batched(ctx, plan, h, dev(np.concatenate([s.y for s in ser])), dev(np.concatenate([s.lnrv for s in ser])),
                        dev(ths), 0.03, minv=minv, seed=4, n_traj=rows, dH_out=dH, accept_out=acc)
    rsv.rsv_sync_status(ctx)
    plan.close()
    return h, dH, acc


@pytest.mark.parametrize("mass", [False, True])
@pytest.mark.parametrize("rho", [0.0, -0.4])
def test_block_shape_leaves_the_bits(mass, rho):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    rsv.rsv_set_leverage(ctx, rho)
    T, n_md = [1, 2, 31, 33, 640, 1000, 7200, 9001], 10
    ths = [(0.9 + 0.01 * i, -0.5, -0.2, 0.05, 0.1) for i in range(len(T))]
    ser = [synth.rsv_series(t, th, seed=i) for i, (t, th) in enumerate(zip(T, ths))]
    minv = dev(np.random.default_rng(5).uniform(0.5, 2.0, sum(T)), torch.float32) if mass else None
    out = [batched(rsv, ctx, T, ths, ser, n_md, s, 3, minv) for s in SHAPES]
    for s, o in zip(SHAPES[1:], out[1:]):
        for a, b in zip(out[0], o):
            assert torch.equal(a, b), s
    ctx.close()


def test_companions_leave_the_bits():
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    r = np.random.default_rng(0)
    first = [700, 3000]
    ths0 = [(0.95, -0.5, -0.2, 0.05, 0.1), (0.9, -0.4, -0.1, 0.06, 0.2)]
    ser0 = [synth.rsv_series(t, th, seed=i) for i, (t, th) in enumerate(zip(first, ths0))]
    out, shapes = [], set()
    for more in ([5], [100] * 300, list(r.integers(2000, 8000, 40))):
        T = first + [int(t) for t in more]
        ths = ths0 + [(0.9, -0.5, -0.2, 0.05, 0.1)] * len(more)
        ser = ser0 + [synth.rsv_series(t, ths[2], seed=9 + i) for i, t in enumerate(T[2:])]
        off = np.concatenate([[0], np.cumsum(T)])
        plan = rsv.Plan(ctx, off, 20, prec="fp64")
        shapes.add((plan.info()["threads"], plan.info()["sites_per_thread"]))
        plan.close()
        h, dH, acc = batched(rsv, ctx, T, ths, ser, 20, None, 3)
        out.append((h[:3700], dH[:, :2], acc[:, :2]))
    assert len(shapes) > 1
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("schedule", [None, (64, 1, 40)])
def test_terms_beyond_the_integer_sum(schedule):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    T, n_md, dtau, th = 300, 2, 1e-9, synth.THETA_STD
    s = synth.rsv_series(T, th, seed=1)
    y = s.y.copy()
    y[[0, 77, 299]] = 1e6, 3e5, 2e9      # y^2/2 e^{-h} up to 1e18
    p0 = synth.standard_normals(T, 2)
    if schedule:
        rsv.rsv_set_schedule(ctx, *schedule)
    h, p = dev(s.h_true), dev(p0)
    dH, _ = rsv.rsv_hmc_trajectory(ctx, h, p, dev(y), dev(s.lnrv), th, n_md, dtau, log_u=dev([-1e300]))
    rsv.rsv_sync_status(ctx)
    h1, p1 = oracle.leapfrog(s.h_true, p0, y, s.lnrv, th, n_md, dtau)
    big = 0.5 * (y * y * np.exp(-s.h_true)).max() + 0.5 * (p1 * p1).max()
    ref = oracle.delta_H(s.h_true, p0, h1, p1, y, s.lnrv, th)
    assert big > 2.0 ** 40 and abs(dH.item() - ref) <= 1e-12 * big
    ctx.close()
