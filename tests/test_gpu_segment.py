"""lj_step_record and lj_vv_adjoint_segment: the states are lj_step's, and the
adjoint over a segment is that of its steps one at a time, here taken in FP64
on the same states."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

pytestmark = pytest.mark.gpu

# (n, density, shift mode, precision, context setting): slotted cells, sorted
# lists (the 27-cell form, deterministic order, a skin), FP64, a cell beyond
# its slots (n = 3 cells a side, dense)
FORMS = [(2048, 0.8442, 2, "mixed", None), (4001, 0.3, 1, "mixed", None), (777, 1.0, 0, "mixed", None),
         (3000, 0.8442, 2, "mixed", "kernel3"), (3000, 0.8442, 1, "mixed", "kernel6"),
         (3000, 0.8442, 2, "mixed", "deterministic"), (3000, 0.8442, 2, "mixed", "skin"),
         (2048, 0.8442, 1, "fp64", None), (2048, 0.8442, 2, "fp64", None)]


@pytest.mark.parametrize("n,rho,mode,precision,setting", FORMS)
@pytest.mark.parametrize("nsteps", [1, 2, 5])
def test_segment_matches_single_steps(n, rho, mode, precision, setting, nsteps):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.lattice_gas(n, rho, 3, 0.05)
    v = inputs.velocities(n, 0.9, 4)

    def system(prec):
        return lj.System(x, v, L, shift_mode=mode, precision=prec)

    s = system(precision)
    if setting in ("kernel3", "kernel6"):
        lj.lj_set_tuning(s.ctx, int(setting[-1]), 0, 4)
    elif setting == "deterministic":
        lj.lj_set_deterministic(s.ctx, True)
    elif setting == "skin":
        lj.lj_set_skin(s.ctx, 0.2, 0)
    s.forces()
    traj = torch.empty((nsteps + 1, n, 3), dtype=torch.float64, device="cuda")
    traj[0].copy_(s.x)
    v1, f1 = s.v.clone(), s.f.clone()
    lj.lj_step_record(s.ctx, traj, v1, f1, nsteps)
    s.check()
    # the same steps in FP64: a force error of RMS 1e-5 F_rms moves positions
    # by at most dt^2 k^2 / 2 of it, velocities by dt k of it
    r = system("fp64")
    r.forces()
    frms = float(r.f[:, :3].pow(2).sum(1).mean().sqrt())
    tol = 1e-5 if precision == "mixed" else 1e-11
    for k in range(1, nsteps + 1):
        r.step(1)
        d = traj[k] - r.x
        d -= L * torch.round(d / L)
        assert float(d.pow(2).mean().sqrt()) <= 0.5 * 0.005 ** 2 * k ** 2 * tol * frms + 1e-13 * L, k
    assert float((v1 - r.v).pow(2).mean().sqrt()) <= 0.005 * nsteps * tol * frms + 1e-13
    assert float((f1[:, :3].double() - r.f[:, :3]).pow(2).sum(1).mean().sqrt()) <= 2 * tol * frms

    g = r.f[:, :3] / frms
    lx, lv = torch.full_like(traj[0], 0.01), g.clone()
    dp = torch.tensor([0.5, -0.25], dtype=torch.float64, device="cuda")
    lj.lj_vv_adjoint_segment(s.ctx, traj, nsteps, lx, lv, dp)
    s.check()
    rx, rv = torch.full_like(traj[0], 0.01), g.clone()
    rp = torch.tensor([0.5, -0.25], dtype=torch.float64, device="cuda")
    for k in range(nsteps - 1, -1, -1):
        lj.lj_vv_adjoint_step(r.ctx, traj[k].contiguous(), traj[k + 1].contiguous(), rx, rv, rp)
    # FP32 pair terms and sums: 1e-5 of the whole (as the VJP's tests); the
    # parameter sums are of one sign here (g along the forces)
    for got, ref in ((lx, rx), (lv, rv), (dp, rp)):
        assert float((got - ref).norm()) <= (1e-5 if precision == "mixed" else 1e-11) * float(ref.norm())
    s.close()
    r.close()
