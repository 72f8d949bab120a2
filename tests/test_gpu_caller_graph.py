"""Calls that a caller records into a CUDA graph of their own: one evaluation
recorded and replayed three times, direct calls before, between and after, in
either state of the count buffers that the slotted binnings alternate, against
the oracle; also recorded as a context's first evaluation, and recorded but
not replayed.  Tolerances: those of the step, force and VJP tests."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import min_image, rel_rms

pytestmark = pytest.mark.gpu


def _record(st, call):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        call()
    return g


def _system(precision, mode, before, seed, n_cells=6):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = inputs.jittered_fcc(n_cells, 0.8442, 0.1, seed)
    v = inputs.velocities(x.shape[0], 0.9, seed)
    st = torch.cuda.Stream()
    s = lj.System(x, v, L, precision=precision, shift_mode=mode, stream=st)
    torch.cuda.synchronize()
    for _ in range(before):
        s.forces()
    torch.cuda.synchronize()
    return s, st, x, v, L


def _cells_match(s, oracle_mod):
    import torch
    from paper_0709_3225_gb300 import lj
    n, ncell = s.n, s.ctx.nc ** 3
    t = [torch.full((k,), -7, dtype=torch.int32, device="cuda") for k in (n, ncell, ncell + 1, n)]
    torch.cuda.synchronize()
    lj.lj_get_cells(s.ctx, *t)
    torch.cuda.synchronize()
    cell_of, count, start, perm = (q.cpu().numpy() for q in t)
    o = oracle_mod.bin_cells(s.x.cpu().numpy(), s.params.box, s.ctx.nc)
    assert np.array_equal(cell_of, o[0]) and np.array_equal(count, o[1]) and np.array_equal(start, o[2])
    assert np.array_equal(np.sort(perm), np.arange(n)) and np.array_equal(cell_of[perm], np.repeat(np.arange(ncell), count))


@pytest.mark.parametrize("precision,mode", [("mixed", 1), ("mixed", 2), ("fp64", 1), ("fp64", 2)])
@pytest.mark.parametrize("before", [0, 1, 2])
def test_forces(oracle_mod, precision, mode, before):
    import torch
    s, st, x, _, L = _system(precision, mode, before, 201)
    tol = 1e-5 if precision == "mixed" else 1e-12
    g = _record(st, lambda: s.forces())
    rng = np.random.default_rng(before)
    for k in range(6):                      # replays and direct calls; the positions change in between
        y = x + rng.normal(0.0, 0.02, x.shape)
        s.x.copy_(torch.as_tensor(y))
        s.f.fill_(float("nan"))
        torch.cuda.synchronize()
        if k in (3, 5):
            s.forces(energy=k == 5)         # FP64 energies: the sorted lists
        else:
            with torch.cuda.stream(st):
                g.replay()
        torch.cuda.synchronize()
        s.check()
        fo = oracle_mod.forces_cells(y, L, mode=mode)[0]
        far = ~oracle_mod.near_cutoff(y, L, band=1e-5 if precision == "mixed" else 1e-12)   # as the force tests
        assert rel_rms(s.f.double().cpu().numpy()[far, :3], fo[far]) <= tol, k
        _cells_match(s, oracle_mod)
    s.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("before,nrec", [(1, 1), (2, 1), (1, 2), (2, 3)])
def test_steps(oracle_mod, precision, before, nrec):
    import torch
    s, st, x, v, L = _system(precision, 2 if precision == "mixed" else 1, before, 202)
    mode = s.params.shift_mode
    xo, vo = x.copy(), v.copy()
    fo = oracle_mod.forces_cells(xo, L, mode=mode)[0]
    g = _record(st, lambda: s.step(nrec))
    done = 0
    for k in ("direct", "replay", "replay", "direct", "replay", "direct", "direct"):
        if k == "direct":
            s.step(1)
            done += 1
            oracle_mod.vv(xo, vo, fo, L, 1, mode=mode)
        else:
            with torch.cuda.stream(st):
                g.replay()
            done += nrec
            oracle_mod.vv(xo, vo, fo, L, nrec, mode=mode)
        torch.cuda.synchronize()
    s.check()
    xt, vt = (2e-6, 2e-4) if precision == "mixed" else (1e-10, 1e-9)
    assert np.abs(min_image(s.x.cpu().numpy() - xo, L)).max() <= xt
    assert np.abs(s.v.cpu().numpy() - vo).max() <= vt
    _cells_match(s, oracle_mod)
    s.close()


def test_langevin_steps():
    """Against the same calls made directly (the random numbers are the same)."""
    import torch
    a, st, x, v, L = _system("mixed", 2, 1, 203)
    b = _system("mixed", 2, 1, 203)[0]
    for s in (a, b):
        s.langevin_seed(11)
    torch.cuda.synchronize()
    g = _record(st, lambda: a.langevin_step(1, 1.0, 0.9))
    for k in range(5):
        if k == 3:
            a.langevin_step(1, 1.0, 0.9)
        else:
            with torch.cuda.stream(st):
                g.replay()
        b.langevin_step(1, 1.0, 0.9)
    torch.cuda.synchronize()
    a.check()
    b.check()
    assert float(np.abs(min_image((a.x - b.x).cpu().numpy(), L)).max()) <= 2e-6
    assert float((a.v - b.v).abs().max()) <= 2e-4
    a.close()
    b.close()


def test_vjp(oracle_mod):
    import torch
    from paper_0709_3225_gb300 import lj
    s, st, x, _, L = _system("mixed", 2, 1, 204, 5)
    gv = np.random.default_rng(204).normal(0.0, 1.0, x.shape)
    gd = torch.as_tensor(gv).cuda()
    dx, dp = torch.zeros_like(s.x), torch.zeros(2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()

    def call():
        lj.lj_forces_vjp(s.ctx, s.x, gd, 1.0, dx, dp)

    call()
    g = _record(st, call)
    for k in range(4):
        if k == 2:
            call()
        else:
            with torch.cuda.stream(st):
                g.replay()
    torch.cuda.synchronize()
    s.check()
    ref = oracle_mod.forces_vjp(x, L, gv, mode=2)
    assert rel_rms(dx.cpu().numpy() / 5.0, ref[0]) <= 1e-5
    for got, want in zip(dp.cpu().numpy() / 5.0, ref[1:]):
        assert abs(got - want) <= 1e-5 * abs(want)
    s.close()


@pytest.mark.parametrize("nrec", [1, 2, 4])
def test_batch_steps(oracle_mod, nrec):
    import torch
    from paper_0709_3225_gb300 import lj
    states = [inputs.jittered_fcc(5, 0.8442, 0.08, 3), inputs.lattice_gas(1999, 0.6, 4, 0.08)]
    xs, boxes = [q[0] for q in states], [q[1] for q in states]
    vs = [inputs.velocities(len(x), 0.8, 20 + i) for i, x in enumerate(xs)]
    st = torch.cuda.Stream()
    b = lj.Batch(xs, vs, boxes, shift_mode=2, stream=st)
    b.set_kernel(7)
    torch.cuda.synchronize()
    b.forces()
    g = _record(st, lambda: b.step(nrec))
    n = 0
    for k in (3, 0, 0, 1, 0, 4):            # direct steps; 0: a replay
        if k:
            b.step(k)
        else:
            with torch.cuda.stream(st):
                g.replay()
        n += k or nrec
    torch.cuda.synchronize()
    b.check()
    x, v = b.x.cpu().numpy(), b.v.cpu().numpy()
    for r in range(b.nrep):
        xo, vo = xs[r].copy(), vs[r].copy()
        fo = oracle_mod.forces_cells(xo, boxes[r], mode=2)[0]
        frms = np.sqrt((fo ** 2).sum(axis=1).mean())
        oracle_mod.vv(xo, vo, fo, boxes[r], n, mode=2)
        # a force error of RMS 1e-5 F_rms over n steps (test_gpu_batch_slots.py)
        d = min_image(b.replica(x, r) - xo, boxes[r])
        assert np.sqrt((d ** 2).mean()) <= 0.5 * 0.005 ** 2 * n ** 2 * 1e-5 * frms, r
        assert np.sqrt(((b.replica(v, r) - vo) ** 2).mean()) <= 0.005 * n * 1e-5 * frms, r
    b.close()


def test_recorded_and_never_replayed(oracle_mod):
    import torch
    s, st, x, _, L = _system("mixed", 1, 0, 205)
    _record(st, lambda: s.forces())
    fo = oracle_mod.forces_cells(x, L, mode=1)[0]
    for _ in range(3):
        s.forces()
        torch.cuda.synchronize()
        s.check()
        assert rel_rms(s.f.double().cpu().numpy()[:, :3], fo) <= 1e-5
        _cells_match(s, oracle_mod)
    s.close()
