"""Batched plans on the planner's block shapes.  A mixed series' results do not
depend on the series it is packed with or the block it lands in: its decisions
and dH are those of the large block bit for bit.  FP64 plans of any shape stay
within the FP64 tolerances of the oracle (1e-12 on h', 1e-9 on dH)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
SETS = {"one": [1], "tiny": [1, 2, 3, 33, 640, 641], "few": [700, 300, 1000, 1280, 999],
        "long": [7680, 12, 2000], "many": list(np.random.default_rng(1).integers(100, 700, 300)),
        "wide": [500, 3000, 6000] * 60}


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def inputs(T, seed=3):
    ths = [(0.9 + 0.001 * (i % 50), -0.5, -0.2, 0.05, 0.1) for i in range(len(T))]
    ser = [synth.rsv_series(int(t), th, seed=seed + i) for i, (t, th) in enumerate(zip(T, ths))]
    off = np.concatenate([[0], np.cumsum(T)])
    return ths, off, np.concatenate([s.h_true for s in ser]), np.concatenate([s.y for s in ser]), np.concatenate([s.lnrv for s in ser])


@pytest.mark.parametrize("name", list(SETS))
@pytest.mark.parametrize("mass", [False, True])
def test_mixed_results_do_not_depend_on_the_block(name, mass):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    T, n_md = SETS[name], 20
    ths, off, h0, y, lr = inputs(T)
    minv = dev(np.random.default_rng(5).uniform(0.5, 2.0, off[-1]), torch.float32) if mass else None
    out = []
    for fixed in (False, True):
        if fixed:
            rsv.rsv_set_schedule(ctx, 384, 20, 384 * 20 - 2 * (n_md + 1) - 3)
        try:
            plan = rsv.Plan(ctx, off, n_md, with_mass=mass)
        finally:
            rsv.rsv_set_schedule(ctx)
        h = dev(h0)
        dH = torch.empty(3, len(T), dtype=torch.float64, device="cuda")
        acc = torch.empty(3, len(T), dtype=torch.int32, device="cuda")
        rsv.rsv_hmc_batched(ctx, plan, h, dev(y), dev(lr), dev(ths), 0.02, minv=minv, seed=4, n_traj=3, dH_out=dH, accept_out=acc)
        rsv.rsv_sync_status(ctx)
        out.append((h, dH, acc))
        plan.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("name", list(SETS))
def test_fp64_against_the_oracle(name):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    T, n_md, dtau = SETS[name], 20, 0.02
    ths, off, h0, y, lr = inputs(T)
    p0 = synth.standard_normals(off[-1], 9)
    plan = rsv.Plan(ctx, off, n_md, prec="fp64")
    h, p = dev(h0), dev(p0)
    dH = torch.empty(len(T), dtype=torch.float64, device="cuda")
    rsv.rsv_hmc_batched(ctx, plan, h, dev(y), dev(lr), dev(ths), dtau, p=p, log_u=dev([-1e300] * len(T)), dH_out=dH)
    rsv.rsv_sync_status(ctx)
    h, dH = h.cpu().numpy(), dH.cpu().numpy()
    for s in range(len(T)):
        a, b = off[s], off[s + 1]
        h1, p1 = oracle.leapfrog(h0[a:b], p0[a:b], y[a:b], lr[a:b], ths[s], n_md, dtau)
        assert np.max(np.abs(h[a:b] - h1) / np.maximum(1.0, np.abs(h1))) <= 1e-12
        assert abs(dH[s] - oracle.delta_H(h0[a:b], p0[a:b], h1, p1, y[a:b], lr[a:b], ths[s])) <= 1e-9
    plan.close()
    ctx.close()


@pytest.mark.parametrize("prec,n_md", [("mixed", 3900), ("fp64", 3600)])
def test_too_many_steps_stay_refused(prec, n_md):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    with pytest.raises(rsv.RSVError, match="RSV_EINVAL"):
        rsv.Plan(ctx, [0, 100, 250], n_md, prec=prec)
    ctx.close()
