"""The FP64 pair-once forces in 64-bit fixed point (the default FP64 forces
without energies, modes 0 and 1) against the oracle: tolerances of the FP64
force tests (1e-12 relative RMS, 1e-10 of the force scale per particle)."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import dense_cluster_state, min_image, rel_rms

pytestmark = pytest.mark.gpu


def _state(name):
    """(x, L, rc, sigma)"""
    if name == "liquid":
        return *inputs.jittered_fcc(8, 0.8442, 0.1, 81), 2.5, 1.0
    if name == "box3":           # 3 cells per side: every image
        return *inputs.jittered_fcc(5, 0.8442, 0.1, 82), 2.5, 1.0
    if name == "cluster":        # cells beyond their slots: the plain path
        return *dense_cluster_state(seed=83), 2.5, 1.0
    if name == "gas":
        return *inputs.lattice_gas(1999, 0.1, 84), 2.5, 1.0
    if name == "images":         # coordinates outside the box
        x, L = inputs.jittered_fcc(6, 0.8442, 0.1, 85)
        return x + L * np.random.default_rng(85).integers(-2, 3, x.shape), L, 2.5, 1.0
    if name == "wca":            # short cutoff, other sigma
        x, L = inputs.jittered_fcc(8, 0.8442, 0.05, 86)
        return x, L, 1.05 * 2.0 ** (1.0 / 6.0), 1.05
    if name == "wide":           # a wide cutoff: cells fuller than the slotted ones take
        x, L = inputs.jittered_fcc(10, 0.3, 0.1, 87)
        return x, L, 4.0, 1.0
    if name == "close":          # pairs far inside the fixed-point range's end
        x, L = inputs.jittered_fcc(6, 0.8442, 0.1, 88)
        x[1] = x[0] + [0.3, 0.0, 0.0]
        x[50] = x[40] + [0.0, 0.5, 0.6]
        x[101] = x[100]          # coincident: no force between them
        return x, L, 2.5, 1.0
    x = np.array([[0.2, 4.0, 4.0], [7.1, 4.0, 4.0], [7.9, 7.9, 7.9]])
    return x, 8.0, 2.5, 1.0


@pytest.mark.parametrize("name", ["liquid", "box3", "cluster", "gas", "images", "wca", "wide", "close", "three"])
@pytest.mark.parametrize("mode", [0, 1])
def test_forces_match_the_oracle(oracle_mod, name, mode):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L, rc, sigma = _state(name)
    s = lj.System(x, None, L, precision="fp64", shift_mode=mode, rc=rc, sigma=sigma, eps=1.3)
    fo = oracle_mod.forces_cells(x, L, mode=mode, rc=rc, sigma=sigma, eps=1.3)[0]
    near = oracle_mod.near_cutoff(x, L, band=1e-12, rc=rc)
    got = []
    for _ in range(2):
        s.f.fill_(float("nan"))
        s.forces()
        got.append(s.f.clone())
    s.check()
    f = got[0].cpu().numpy()
    s.close()
    assert np.all(f[:, 3] == 0.0)
    f = f[:, :3]
    assert np.all(np.isfinite(f))
    good = np.isfinite(fo).all(axis=1)   # the oracle's force of coincident particles is no number
    assert good.sum() >= x.shape[0] - 2
    f, fo, near = f[good], fo[good], near[good]
    # integer sums: the same bits whatever the order (but for the pairs taken
    # in FP64, and for "wide", whose 32 particles a cell take the sorted lists)
    if name not in ("close", "cluster", "wide"):
        assert torch.equal(got[0], got[1])
    assert rel_rms(f, fo) <= 1e-12
    scale = np.abs(fo).max(axis=1) + np.sqrt((fo ** 2).sum(axis=1).mean()) * (name != "close")
    assert np.all(np.abs(f - fo).max(axis=1)[~near] <= 1e-10 * (scale + 1.0)[~near])


@pytest.mark.parametrize("graph", [False, True])
def test_steps_follow_the_oracle(oracle_mod, graph):
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(8, 0.8442, 0.1, 89)
    v = inputs.velocities(x.shape[0], 0.9, 89)
    xo, vo = x.copy(), v.copy()
    fo = oracle_mod.forces_cells(xo, L, mode=1)[0]
    s = lj.System(x, v, L, precision="fp64")
    lj.lj_set_graph(s.ctx, graph)
    for n in (1, 6, 7):
        s.step(n)
        oracle_mod.vv(xo, vo, fo, L, n, mode=1)
        assert np.abs(min_image(s.x.cpu().numpy() - xo, L)).max() <= 1e-10
        assert np.abs(s.v.cpu().numpy() - vo).max() <= 1e-9
        # f is the whole force after every call: an energy evaluation in between
        e = s.energy()
        assert rel_rms(s.f.cpu().numpy()[:, :3], oracle_mod.forces_cells(s.x.cpu().numpy(), L, mode=1)[0]) <= 1e-11
    s.check()
    s.close()


def test_host_steps_and_lists(oracle_mod):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(12, 0.8442, 0.1, 90)   # 6,912 particles: copied in four parts
    v = inputs.velocities(x.shape[0], 0.9, 90)
    a = lj.System(x, v, L, precision="fp64")
    a.forces()
    xh, vh, fh = (t.cpu().pin_memory() for t in (a.x, a.v, a.f))
    a.step(2)
    lj.lj_step_host(a.ctx, xh, vh, fh, 2)
    assert torch.equal(xh, a.x.cpu()) and torch.equal(vh, a.v.cpu()) and torch.equal(fh, a.f.cpu())
    ncell = a.ctx.nc ** 3
    t = [torch.empty(k, dtype=torch.int32, device="cuda") for k in (a.n, ncell, ncell + 1, a.n)]
    lj.lj_get_cells(a.ctx, *t)
    cell_of, count, start, perm = (q.cpu().numpy() for q in t)
    o = oracle_mod.bin_cells(a.x.cpu().numpy(), L, a.ctx.nc)
    assert np.array_equal(cell_of, o[0]) and np.array_equal(count, o[1]) and np.array_equal(start, o[2])
    assert np.array_equal(np.sort(perm), np.arange(a.n)) and np.array_equal(cell_of[perm], np.repeat(np.arange(ncell), count))
    a.check()
    a.close()
