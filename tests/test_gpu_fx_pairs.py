"""FP64 forces of single pairs, near and far: relative to each pair's own
force, against the pair law in extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 1.3


def _pairs(L, r, seed):
    """Isolated pairs at distance r, one per 10^3 of space, anywhere in it (also across the box's faces)."""
    rng = np.random.default_rng(seed)
    m = int(L // 10)
    g = np.stack(np.meshgrid(*[np.arange(m) * (L / m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    a = g + rng.uniform(-1.0, 1.0, g.shape)
    u = rng.normal(size=g.shape)
    b = a + r * u / np.linalg.norm(u, axis=1)[:, None]
    x = np.empty((2 * len(a), 3))
    x[0::2], x[1::2] = a, b
    x -= L * np.floor(x / L)
    x[x >= L] -= L
    return x


def _exact(x, L, sigma):
    """F on the first of each pair: the law in long double on the given coordinates."""
    d = x[0::2].astype(np.longdouble) - x[1::2].astype(np.longdouble)
    d -= np.longdouble(L) * np.round((d / np.longdouble(L)).astype(np.float64))
    u = np.longdouble(sigma) ** 2 / (d * d).sum(1)
    return (24 * np.longdouble(EPS) / np.longdouble(sigma) ** 2 * u ** 4 * (2 * u ** 3 - 1))[:, None] * d


@pytest.mark.parametrize("rc,sigma", [(2.5, 1.0), (2.6, 1.0), (2.5, 1.05), (1.7, 1.0), (3.0, 1.0), (4.0, 1.0)])
@pytest.mark.parametrize("r", [0.8, 0.93, 1.0, 1.1, 1.2, 1.5, 1.79, 1.81, 2.0, 2.2, 2.45, 2.9, 3.9])
def test_relative_error_of_single_pairs(rc, sigma, r):
    import torch
    from paper_0709_3225_gb300 import lj
    if r >= rc:
        pytest.skip("out of range")
    for L in (21.3, 30.7):   # (a larger, emptier box keeps the sorted lists and FP64)
        x = _pairs(L, r, int(1000 * r + L))
        s = lj.System(x, None, L, precision="fp64", rc=rc, sigma=sigma, eps=EPS)
        s.forces()
        s.check()
        f = s.f[:, :3].cpu().numpy()
        s.close()
        want = _exact(x, L, sigma)
        norm = np.sqrt((want * want).sum(1)).astype(np.float64)
        err = np.sqrt(((f[0::2] - want) ** 2).sum(1)).astype(np.float64)
        v = r / sigma
        if rc > 2.6 * sigma or v * v < 0.8:
            # FP64 coordinates, the cells' centres and the image shift rounded at the scale of L
            # (4 roundings of at most ulp(L) / 2 in each of 3 components), a force that goes as r^-14 at most
            tol = (14.0 / r) * np.sqrt(3.0) * 2.0 * np.spacing(L) * np.maximum(norm, 24 * EPS / sigma * v ** -13)
        else:
            assert np.array_equal(f[0::2], -f[1::2])
            # half a unit in each of the three components, and 5 roundings of 2^-53
            unit = 24 * EPS / sigma * 2.0 ** -52 / (1 if v < 2 ** (1 / 6) else 32 if v < 1.8 else 256)
            tol = np.sqrt(3.0) / 2.0 * unit * max(1.0, sigma) * 2.0 ** (sigma != 1.0) + 5.0 * 2.0 ** -53 * norm
        assert np.all(err <= tol), float((err / tol).max())
