"""The batch's pair-once kernel on slotted cells: replicas of uneven size and
density, with cells beyond their slots, three cells a side and non-finite
particles, against the oracle; step counts that leave the count buffers in
either state, replayed and direct; the kernel changed in between."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import dense_cluster_state, min_image, rel_rms

pytestmark = pytest.mark.gpu


def _replicas():
    states = [inputs.jittered_fcc(5, 0.8442, 0.08, 3), inputs.lattice_gas(1999, 0.6, 4, 0.08),
              dense_cluster_state(seed=5), inputs.lattice_gas(3001, 0.9, 6, 0.05),
              inputs.lattice_gas(417, 0.95, 7, 0.05)]
    return [s[0] for s in states], [s[1] for s in states]


@pytest.mark.parametrize("mode,energy", [(0, False), (1, True), (2, False), (2, True)])
def test_forces_of_uneven_replicas(oracle_mod, mode, energy):
    from paper_0709_3225_gb300 import lj
    xs, boxes = _replicas()
    vs = [np.zeros_like(x) for x in xs]
    b = lj.Batch(xs, vs, boxes, shift_mode=mode)
    b.set_kernel(7)
    for _ in range(3):                      # both count buffers
        b.forces(energy=energy)
    b.check()
    f = b.f.double().cpu().numpy()
    for r in range(b.nrep):
        fo, epo, _, _ = oracle_mod.forces_cells(xs[r], boxes[r], mode=mode)
        assert rel_rms(b.replica(f, r)[:, :3], fo) <= 1e-5, r
        if energy:
            assert np.abs(b.replica(f, r)[:, 3] - epo).max() <= 1e-5 * np.abs(epo).max(), r
    b.close()


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("counts", [(1, 2, 3, 4), (5, 1, 6), (3, 3, 2, 4)])
def test_steps_in_either_buffer(oracle_mod, use_graph, counts):
    from paper_0709_3225_gb300 import lj
    xs, boxes = _replicas()
    xs, boxes = xs[:2] + xs[3:], boxes[:2] + boxes[3:]
    vs = [inputs.velocities(x.shape[0], 0.8, 20 + i) for i, x in enumerate(xs)]
    b = lj.Batch(xs, vs, boxes, shift_mode=2)
    b.set_kernel(7)
    b.set_tuning(cells_per_grab=2, use_graph=use_graph)
    b.forces()
    for k, c in enumerate(counts):
        b.step(c)
        if k == 1:                          # the 27-cell code in between
            b.set_kernel(3)
            b.forces()
            b.set_kernel(7)
    b.check()
    assert b.launches()[1] == (use_graph and max(counts[2:]) >= 3)
    n = sum(counts)
    x = b.x.cpu().numpy()
    v = b.v.cpu().numpy()
    for r in range(b.nrep):
        xo, vo = xs[r].copy(), vs[r].copy()
        fo = oracle_mod.forces_cells(xo, boxes[r], mode=2)[0]
        frms = np.sqrt((fo ** 2).sum(axis=1).mean())
        oracle_mod.vv(xo, vo, fo, boxes[r], n, mode=2)
        # a force error of RMS 1e-5 F_rms over n steps: dt^2 n^2 / 2 of it in x, dt n in v
        d = min_image(b.replica(x, r) - xo, boxes[r])
        assert np.sqrt((d ** 2).mean()) <= 0.5 * 0.005 ** 2 * n ** 2 * 1e-5 * frms, r
        assert np.sqrt(((b.replica(v, r) - vo) ** 2).mean()) <= 0.005 * n * 1e-5 * frms, r
    b.close()


def test_non_finite_particles_leave_the_others(oracle_mod):
    from paper_0709_3225_gb300 import lj
    xs, boxes = _replicas()
    b = lj.Batch(xs, [np.zeros_like(x) for x in xs], boxes)
    b.set_kernel(7)
    b.x[0, 0] = float("nan")
    b.x[b.offsets[3] + 5, 2] = float("inf")
    for _ in range(2):
        b.forces()
        with pytest.raises(lj.LJError) as ei:
            b.check()
        assert ei.value.code == lj.LJ_ENONFINITE
        f = b.f.double().cpu().numpy()
        for r, bad in ((0, [0]), (3, [5]), (1, [])):
            good = np.setdiff1d(np.arange(len(xs[r])), bad)
            fo = oracle_mod.forces_cells(np.ascontiguousarray(xs[r][good]), boxes[r], mode=1)[0]
            assert rel_rms(b.replica(f, r)[good, :3], fo) <= 1e-5, r
    b.close()
