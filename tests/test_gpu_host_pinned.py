"""lj_step_host on pinned arrays (read and written by the kernels in place):
the same as lj_step on device arrays at the edges of blocks and of the size
below which x goes back with v and f; and as on pageable arrays and on pinned
ones that are not 16-byte aligned, which are copied."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 255, 256, 257, 4097, 32768, 32769, 70001])
@pytest.mark.parametrize("steps,memory", [(1, "pinned"), (2, "pinned"), (3, "pageable"), (3, "pinned"), (2, "offset")])
def test_host_steps_match_device_steps(n, steps, memory):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.lattice_gas(n, 0.6 if n > 1000 else 0.3 if n > 200 else 0.004, 5, 0.05)
    v = inputs.velocities(n, 0.9, 6)
    s = lj.System(x, v, L, shift_mode=2)
    s.forces()
    s.check()

    def host(t):
        if memory == "pageable":
            return t.cpu().clone()
        if memory == "pinned":
            return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
        k = 8 // t.element_size()
        return torch.empty(t.numel() + k, dtype=t.dtype, pin_memory=True)[k:].view(t.shape).copy_(t)

    for call in range(2):                    # both count buffers
        hx, hv, hf = host(s.x), host(s.v), host(s.f)
        lj.lj_step_host(s.ctx, hx, hv, hf, steps)
        s.step(steps)
        s.check()
        frms = float(s.f[:, :3].double().pow(2).sum(1).mean().sqrt())
        # two evaluations differ by the order of FP32 sums, 1e-6 of F_rms:
        # dt^2 k^2 / 2 of it in x, dt k in v
        d = hx - s.x.cpu()
        d -= L * torch.round(d / L)
        assert float(d.pow(2).mean().sqrt()) <= 0.5 * (0.005 * steps) ** 2 * 1e-6 * frms + 1e-14 * L
        assert float((hv - s.v.cpu()).pow(2).mean().sqrt()) <= 0.005 * steps * 1e-6 * frms + 1e-15
        assert float((hf[:, :3] - s.f[:, :3].cpu()).double().pow(2).sum(1).mean().sqrt()) <= 2e-6 * frms + 1e-30
    s.close()


def test_host_step_reports_non_finite():
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.lattice_gas(1000, 0.5, 7, 0.05)
    s = lj.System(x, np.zeros_like(x), L)
    s.forces()
    a = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (s.x, s.v, s.f)]
    a[0][17, 1] = float("nan")
    with pytest.raises(lj.LJError) as ei:
        lj.lj_step_host(s.ctx, *a, 1)
    assert ei.value.code == lj.LJ_ENONFINITE
    s.close()
