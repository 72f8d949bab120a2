"""The first gradient on a small context allocates no more than the second
(its cotangents' slots came with the context), but for its accumulator."""
import time

import pytest

from paper_0709_3225_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_first_gradient_takes_little_longer_than_the_second():
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(20, 0.8442, 0.05, 91)
    t = ([], [])
    for _ in range(12):
        s = lj.System(x, None, L, shift_mode=2)
        s.forces()
        g, dx = torch.ones_like(s.x), torch.zeros_like(s.x)
        dp = torch.zeros(2, dtype=torch.float64, device="cuda")
        for k in range(2):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lj.lj_forces_vjp(s.ctx, s.x, g, 1.0, dx, dp)
            torch.cuda.synchronize()
            t[k].append(time.perf_counter() - t0)
        s.close()
    first, second = (sorted(v)[len(v) // 2] for v in t)
    # 32,000 particles: 143 us against 45 when the slots were allocated here, 61 now; one
    # allocation of their size takes some 90 us
    assert first - second <= 50e-6
