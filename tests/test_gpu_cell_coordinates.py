"""The FP32 coordinates that the force kernels work on are float32(x - c), c
the centre of x's cell, rounded once: with x - c within a few last places of x
of the middle between two floats, particles moved to the double next to c +
float32(x - c) have bit for bit the same forces.  The states are pairs alone in
every third cell, so that a force is one pair term and no order of summation
shows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RC, NC, L = 2.5, 12, 30.37


def _pairs(seed):
    rng = np.random.default_rng(seed)
    cw = L / NC
    k = np.arange(1, NC, 3)   # (in cell 0 the subtraction in FP64 is not exact)
    cell = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    c = (cell + 0.5) * cw
    d = rng.standard_normal(c.shape)
    d *= rng.uniform(0.95, 1.8, (len(c), 1)) / np.linalg.norm(d, axis=1, keepdims=True)
    mid = rng.uniform(-0.25, 0.25, c.shape)
    r = np.stack([mid + 0.5 * d, mid - 0.5 * d], 1).astype(np.float32)
    c = np.repeat(c[:, None], 2, 1)
    x = c + (r.astype(np.float64) + 0.5 * np.spacing(r).astype(np.float64))
    x += rng.integers(-4, 5, x.shape) * np.spacing(x)
    moved = c + (x - c).astype(np.float32).astype(np.float64)
    assert np.array_equal((moved - c).astype(np.float32), (x - c).astype(np.float32))
    return x.reshape(-1, 3), moved.reshape(-1, 3)


def _forces(x, path):
    from paper_0709_3225_gb300 import lj
    if path == "batch":
        b = lj.Batch([x], [np.zeros_like(x)], [L], rc=RC)
        b.set_kernel(7)
        b.forces()
        b.check()
        f = b.f.cpu().numpy()
        b.close()
        return f
    s = lj.System(x, None, L, rc=RC)
    assert s.ctx.nc == NC
    if path == "lists":
        lj.lj_set_tuning(s.ctx, 3)
    s.forces()
    s.check()
    f = s.f.cpu().numpy()
    s.close()
    return f


@pytest.mark.parametrize("path", ["slots", "lists", "batch"])
def test_coordinates_are_rounded_once(path):
    for seed in range(8):
        x, moved = _pairs(seed)
        f, g = _forces(x, path), _forces(moved, path)
        assert np.all(np.abs(f[:, :3]).max(axis=1) > 0)
        assert np.array_equal(f[:, :3], g[:, :3])
