"""With leverage (and in FP64) the block shape of a chain is the one of
rsv_hmc_trajectory and rsv_set_persistent does not reach it: the same results
bit for bit, dH included.  And the shape follows the number of steps: at 2^20
sites few steps take the shorter runs, whose energies cost less."""
import numpy as np
import pytest
import torch

from paper_1603_08114_gb300 import synth

pytestmark = pytest.mark.gpu
TH, RHO = synth.THETA_STD, synth.RHO_STD


def dev(a, dtype=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("T", [700, 20011, 100003, 700001])
@pytest.mark.parametrize("prec,rho", [("mixed", RHO), ("fp64", RHO), ("fp64", 0.0)])
@pytest.mark.parametrize("mass", [False, True])
def test_chain_trajectory_and_switch_agree(T, prec, rho, mass):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    rsv.rsv_set_leverage(ctx, rho)
    s = synth.rsv_series_leverage(T, TH, RHO, seed=T)
    y, lr, th = dev(s.y), dev(s.lnrv), dev(TH)
    minv = dev(np.random.default_rng(1).uniform(0.5, 2.0, T), torch.float32) if mass else None
    n_md, dtau = 12, 0.02
    h1 = dev(s.h_true)
    dH1, acc1 = rsv.rsv_hmc_trajectory(ctx, h1, None, y, lr, TH, n_md, dtau, prec=prec, minv=minv, seed=3, traj=7)
    shapes, out = [], []
    for on in (True, False):
        rsv.rsv_set_persistent(ctx, on)
        cs = rsv.rsv_chain_schedule(ctx, T, n_md, prec, with_mass=mass)
        shapes.append((cs["threads"], cs["sites_per_thread"], cs["tile"]))
        for n in (1, 3):
            h, dH = dev(s.h_true), torch.empty(n, dtype=torch.float64, device="cuda")
            acc = torch.empty(n, dtype=torch.int32, device="cuda")
            rsv.rsv_hmc_chain(ctx, h, y, lr, th, n_md, dtau, n, prec=prec, minv=minv, seed=3, traj0=7, dH_out=dH, accept_out=acc)
            out.append((h, dH, acc))
    rsv.rsv_sync_status(ctx)
    assert shapes[0] == shapes[1]
    for a, b in zip(out[1], out[3]):
        assert torch.equal(a, b)
    for k in (0, 2):
        assert torch.equal(out[k][1], dH1) and torch.equal(out[k][2], acc1)
        if acc1.item():  # (a mixed chain writes a rejected state back as its (hi, lo) pair)
            assert torch.equal(out[k][0], h1)
    ctx.close()


@pytest.mark.parametrize("n_md,j", [(8, 12), (100, 20)])
def test_shape_follows_the_number_of_steps(n_md, j):
    from paper_1603_08114_gb300 import rsv
    ctx = rsv.Context(0)
    rsv.rsv_set_leverage(ctx, RHO)
    assert rsv.rsv_chain_schedule(ctx, 1 << 20, n_md, "mixed")["sites_per_thread"] == j
    ctx.close()
