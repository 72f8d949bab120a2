"""All-pairs forces with groups of particles left out by their bounding boxes:
particles in lattice order, shuffled, in clumps across the boundary, and one
non-finite, at sizes around the groups of 32, against the oracle."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import rel_rms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rho", [(31, 0.02), (33, 0.02), (1000, 0.1), (2047, 0.5), (8200, 0.8442)])
@pytest.mark.parametrize("order", ["lattice", "shuffled", "moved"])
@pytest.mark.parametrize("energy", [False, True])
def test_orders(oracle_mod, n, rho, order, energy):
    from paper_0709_3225_gb300 import lj
    x, L = inputs.lattice_gas(n, rho, 9, 0.05)
    if order == "shuffled":
        x = np.ascontiguousarray(x[np.random.default_rng(1).permutation(n)])
    elif order == "moved":
        x = np.ascontiguousarray((x + np.array([0.37, 0.81, 0.55]) * L) % L)
    s = lj.System(x, None, L, shift_mode=2)
    r = lj.lj_forces_n2(s.ctx, s.x, s.f, energy=energy)
    s.check()
    # per particle, the bound of this kernel's coordinates (test_gpu_n2.py);
    # energies: the same 2e-6 and 1e-4, and the rounding of the shifts (0.1 for
    # a pair, 2^-24 of it), which is what is left of a pair near rc
    fo, ep, e, w = oracle_mod.forces_cells(x, L, mode=2)
    K, S = oracle_mod.stiffness(x, L, mode=2)
    near = oracle_mod.near_cutoff(x, L, band=1e-5)
    f = s.f.double().cpu().numpy()
    d = np.abs(f[:, :3] - fo).max(axis=1)
    dr = 3 * 2.0 ** -25 * L + 2.0 ** -24 * 2.5
    # (1e-7: the rounding of F(rc), 0.039, against which the force of a pair
    # near rc cancels)
    assert np.all(d[~near] <= (1.5 * dr * K + 1e-5 * S + 1e-7)[~near])
    if energy:
        assert abs(r[0] - e) <= 2e-6 * np.abs(ep).sum() + 1e-7 * n
        assert np.abs(f[:, 3] - ep)[~near].max() <= 1e-4 * np.abs(ep).max() + 1e-7
    s.close()


def test_non_finite_particle_leaves_the_others(oracle_mod):
    from paper_0709_3225_gb300 import lj
    x, L = inputs.lattice_gas(1500, 0.3, 11, 0.05)
    bad = [40, 1499]
    good = np.setdiff1d(np.arange(1500), bad)
    fo = oracle_mod.forces_cells(np.ascontiguousarray(x[good]), L, mode=1)[0]
    x[40, 1], x[1499, 0] = np.nan, np.inf
    s = lj.System(x, None, L)
    lj.lj_forces_n2(s.ctx, s.x, s.f)
    with pytest.raises(lj.LJError) as ei:
        s.check()
    assert ei.value.code == lj.LJ_ENONFINITE
    assert rel_rms(s.f.double().cpu().numpy()[good, :3], fo) <= 1e-5
    s.close()
