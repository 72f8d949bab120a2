"""torch.autograd wrappers over the library's forces and their adjoint.

``forces(x, theta, ctx)``  -> F (n, 3) float64; backward gives dL/dx and
                              dL/dtheta, theta = (eps, sigma).
``trajectory(x0, v0, theta, ctx, nsteps, every)`` -> (x_T, v_T) after nsteps
                              velocity-Verlet steps; backward runs the adjoint
                              with checkpoints every ``every`` steps.

The paper has no adjoint; these differentiate its force (Eq. n2_force with the
Section 2 pair force, rc held fixed) and its velocity-Verlet integration.
The cell list is piecewise constant and contributes no derivative.  Every
arithmetic step runs in the library's kernels (lj_forces, lj_step,
lj_forces_vjp, lj_step_record, lj_vv_adjoint_segment); this module only sequences the calls and
keeps checkpoints.  Use the force-shifted potential (shift_mode 2) when the
trajectory derivative must match finite differences: with the energy shift
the force jumps at rc and the trajectory is not differentiable there.
"""
from __future__ import annotations

import torch

from . import lj


def _set(ctx: lj.Context, theta: torch.Tensor) -> torch.Tensor:
    """Give the context theta; returns it in host memory, for the backward
    pass (one read of both values, and none there: the gradient of a force
    misfit at 32,000 particles, whose time is the calls, 598 -> 560 us)."""
    host = theta.detach().to("cpu")
    t = host.tolist()
    if isinstance(t[0], list):
        t = [float(host[0]), float(host[1])]
    lj.lj_set_params(ctx, t[0], t[1])
    return host


def _set_again(ctx: lj.Context, theta: torch.Tensor, host: torch.Tensor) -> None:
    """The same in the backward pass, without a wait for the device where the
    context works on the current stream (otherwise the read of theta orders
    the two streams)."""
    if ctx.stream_ptr == lj._stream_ptr(None):
        _set(ctx, host)
    else:
        _set(ctx, theta)


class _Forces(torch.autograd.Function):
    @staticmethod
    def forward(fctx, x, theta, ctx):
        host = _set(ctx, theta)
        f = torch.empty((ctx.n, 4), dtype=ctx.force_dtype, device=x.device)
        lj.lj_forces(ctx, x.detach().contiguous(), f)
        fctx.ctx = ctx
        fctx.save_for_backward(x.detach(), theta.detach(), host)
        return f[:, :3].to(torch.float64)

    @staticmethod
    def backward(fctx, g):
        x, theta, host = fctx.saved_tensors
        ctx = fctx.ctx
        _set_again(ctx, theta, host)
        dx = torch.zeros_like(x)
        dp = torch.zeros(2, dtype=torch.float64, device=x.device)
        lj.lj_forces_vjp(ctx, x, g.to(torch.float64).contiguous(), 1.0, dx, dp)
        return dx, dp.to(theta.device, theta.dtype), None


class _Trajectory(torch.autograd.Function):
    @staticmethod
    def forward(fctx, x0, v0, theta, ctx, nsteps, every):
        host = _set(ctx, theta)
        x = x0.detach().clone().contiguous()
        v = v0.detach().clone().contiguous()
        f = torch.empty((ctx.n, 4), dtype=ctx.force_dtype, device=x.device)
        lj.lj_forces(ctx, x, f)
        ckpts = []
        done = 0
        while done < nsteps:
            k = min(every, nsteps - done)
            ckpts.append((x.clone(), v.clone(), k))
            lj.lj_step(ctx, x, v, f, k)
            done += k
        fctx.ctx = ctx
        fctx.ckpts = ckpts
        fctx.save_for_backward(theta.detach(), host)
        return x, v

    @staticmethod
    def backward(fctx, gx, gv):
        theta, host = fctx.saved_tensors
        ctx = fctx.ctx
        _set_again(ctx, theta, host)
        ref = fctx.ckpts[0][0]
        lam_x = torch.zeros_like(ref) if gx is None else gx.to(torch.float64).clone().contiguous()
        lam_v = torch.zeros_like(ref) if gv is None else gv.to(torch.float64).clone().contiguous()
        dp = torch.zeros(2, dtype=torch.float64, device=ref.device)
        f = torch.empty((ctx.n, 4), dtype=ctx.force_dtype, device=ref.device)
        for xs, vs, k in reversed(fctx.ckpts):
            # recompute the segment's states from its checkpoint
            traj = torch.empty((k + 1, ctx.n, 3), dtype=torch.float64, device=xs.device)
            traj[0].copy_(xs)
            v = vs.clone()
            lj.lj_forces(ctx, traj[0], f)
            lj.lj_step_record(ctx, traj, v, f, k)
            lj.lj_vv_adjoint_segment(ctx, traj, k, lam_x, lam_v, dp)
        fctx.ckpts = None
        return lam_x, lam_v, dp.to(theta.device, theta.dtype), None, None, None


def forces(x: torch.Tensor, theta: torch.Tensor, ctx: lj.Context) -> torch.Tensor:
    """Differentiable forces F(x; eps, sigma) (n, 3) float64."""
    return _Forces.apply(x, theta, ctx)


def trajectory(x0: torch.Tensor, v0: torch.Tensor, theta: torch.Tensor, ctx: lj.Context, nsteps: int,
               every: int = 10):
    """Differentiable (x_T, v_T) after nsteps velocity-Verlet steps from
    (x0, v0); the backward pass recomputes each segment of ``every`` steps
    from its checkpoint."""
    return _Trajectory.apply(x0, v0, theta, ctx, int(nsteps), int(every))
