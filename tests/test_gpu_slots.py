"""Slotted cells (the binning of the default FP32-mixed path): after forces,
steps and VJPs lj_get_cells returns the lists of the last binning, exactly the
oracle's, with cells beyond their slots and non-finite particles; calls that
need the sorted lists can come in between; graph replay in pairs of steps."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import dense_cluster_state, min_image, rel_rms

pytestmark = pytest.mark.gpu


def _lists(s):
    import torch
    from paper_0709_3225_gb300 import lj
    n, ncell = s.n, s.ctx.nc ** 3
    a = [torch.full((k,), -7, dtype=torch.int32, device="cuda") for k in (n, ncell, ncell + 1, n)]
    lj.lj_get_cells(s.ctx, *a)
    return [t.cpu().numpy() for t in a]


def _check_lists(s, oracle_mod, good=None):
    cell_of, count, start, perm = _lists(s)
    x = s.x.cpu().numpy()
    good = np.ones(s.n, bool) if good is None else good
    idx = np.flatnonzero(good)
    o_cell, o_count, o_start, o_perm = oracle_mod.bin_cells(np.ascontiguousarray(x[good]), s.params.box, s.ctx.nc)
    assert np.array_equal(cell_of[good], o_cell) and np.all(cell_of[~good] == s.ctx.nc ** 3)
    assert np.array_equal(count, o_count) and np.array_equal(start, o_start)
    assert np.array_equal(np.sort(perm), np.arange(s.n))
    assert np.array_equal(np.sort(perm[len(idx):]), np.flatnonzero(~good))
    order = np.lexsort((perm[:len(idx)], cell_of[perm[:len(idx)]]))
    assert np.array_equal(perm[:len(idx)][order], idx[o_perm])


@pytest.mark.parametrize("state", ["liquid", "cluster", "box3", "gas", "three"])
def test_lists_after_forces_steps_and_vjp(oracle_mod, state):
    import torch
    from paper_0709_3225_gb300 import lj
    if state == "liquid":
        x, L = inputs.jittered_fcc(9, 0.8442, 0.1, 71)
    elif state == "cluster":
        x, L = dense_cluster_state(seed=72)          # cells beyond their slots
    elif state == "box3":
        x, L = inputs.jittered_fcc(5, 0.8442, 0.1, 73)
    elif state == "gas":
        x, L = inputs.lattice_gas(1999, 0.1, 74)
    else:
        x, L = inputs.lattice_gas(3, 0.005, 75)
    v = inputs.velocities(x.shape[0], 0.7, 76)
    s = lj.System(x, v, L, dt=0.001, shift_mode=2)
    s.forces()
    _check_lists(s, oracle_mod)
    s.step(3)
    _check_lists(s, oracle_mod)
    lj.lj_bin(s.ctx, s.x)                            # the sorted lists in between
    _check_lists(s, oracle_mod)
    s.langevin_seed(5)
    s.langevin_step(2, 1.0, 0.7)
    _check_lists(s, oracle_mod)
    g = torch.ones_like(s.x)
    lj.lj_forces_vjp(s.ctx, s.x, g, 1.0, torch.zeros_like(s.x), torch.zeros(2, dtype=torch.float64, device="cuda"))
    _check_lists(s, oracle_mod)
    f0 = s.f.clone()
    s.forces()
    s.check()
    assert rel_rms(s.f.double().cpu().numpy(), f0.double().cpu().numpy()) <= 1e-6
    s.close()


def test_lists_with_non_finite_particles(oracle_mod):
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(8, 0.8442, 0.1, 77)
    bad = np.array([0, 31, 700, 2047])
    x[bad, [0, 1, 2, 0]] = [np.nan, np.inf, -np.inf, np.nan]
    s = lj.System(x, None, L)
    good = np.isfinite(x).all(axis=1)
    for _ in range(2):
        s.forces()
        _check_lists(s, oracle_mod, good)
    with pytest.raises(lj.LJError) as ei:
        s.check()
    assert ei.value.code == lj.LJ_ENONFINITE
    s.close()


@pytest.mark.parametrize("counts", [(3, 4, 5, 8), (7, 1, 6, 6), (2, 4, 10, 4)])
def test_graph_replay_in_pairs(oracle_mod, counts):
    """Step counts that leave the count buffers in either state between
    calls, and a call on the sorted lists between two captured ones."""
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(8, 0.8442, 0.1, 78)
    v = inputs.velocities(x.shape[0], 0.7, 78)
    xo, vo = x.copy(), v.copy()
    fo = oracle_mod.forces_cells(xo, L, mode=2)[0]
    oracle_mod.vv(xo, vo, fo, L, sum(counts), mode=2)
    s = lj.System(x, v, L, shift_mode=2)
    lj.lj_set_graph(s.ctx)
    for k, c in enumerate(counts):
        s.step(c)
        if k == 1:
            lj.lj_set_deterministic(s.ctx, True)
            s.forces()
            lj.lj_set_deterministic(s.ctx, False)
    s.check()
    _check_lists(s, oracle_mod)
    assert np.abs(min_image(s.x.cpu().numpy() - xo, L)).max() <= 2e-6
    assert np.abs(s.v.cpu().numpy() - vo).max() <= 2e-4
    s.close()
