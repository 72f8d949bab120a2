"""Liquid droplets in boxes whose mean density is a vapour's: their cells have
slots (no plain path around them), and the FP64 kernel takes the candidates
that do not fit a warp's slice in parts."""
import numpy as np
import pytest

from paper_0709_3225_gb300 import inputs

from gpu_util import min_image, rel_rms

pytestmark = pytest.mark.gpu


def _droplet(m, rho, seed, shift=0.5):
    x, L0 = inputs.jittered_fcc(m, 0.8442, 0.08, seed)
    L = (x.shape[0] / rho) ** (1.0 / 3.0)
    return x + shift * (L - L0), L


# 1.01: across the box's faces; rc 1.2: cells of a few particles
@pytest.mark.parametrize("m,rho,shift,rc", [(8, 0.1, 0.5, 2.5), (8, 0.1, 1.01, 2.5), (7, 0.2, 0.5, 2.5), (9, 0.3, 0.37, 2.5),
                                            (8, 0.5, 0.5, 2.5), (6, 0.15, 0.5, 2.6), (8, 0.2, 0.5, 1.2)])
@pytest.mark.parametrize("mode", [0, 1])
def test_fp64_forces(oracle_mod, m, rho, shift, rc, mode):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = _droplet(m, rho, 31, shift)
    s = lj.System(x, None, L, precision="fp64", shift_mode=mode, rc=rc)
    got = []
    for _ in range(3):
        s.f.fill_(float("nan"))
        s.forces()
        got.append(s.f.clone())
    s.check()
    s.close()
    fo = oracle_mod.forces_cells(x, L, mode=mode, rc=rc)[0]
    assert rel_rms(got[0].cpu().numpy()[:, :3], fo) <= 1e-12
    # integer sums throughout: the plain path's FP64 adds would depend on their order
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


def test_fp64_steps(oracle_mod):
    from paper_0709_3225_gb300 import lj
    x, L = _droplet(8, 0.1, 32)
    v = inputs.velocities(x.shape[0], 0.7, 32)
    s = lj.System(x, v, L, precision="fp64")
    s.step(7)
    s.check()
    fo = oracle_mod.forces_cells(x, L, mode=1)[0]
    oracle_mod.vv(x, v, fo, L, 7, mode=1)
    assert np.abs(min_image(s.x.cpu().numpy() - x, L)).max() <= 1e-10
    s.close()


def _time(fn):
    import torch
    best = 1e9
    for _ in range(12):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


# per call, droplet at 0.1 against a liquid of as many particles: VJP 324 us and
# 27 with 16 slots a cell, FP64 1,030 and 37 with no parts; 52 and 27, 60 and 37 now
@pytest.mark.parametrize("what", ["vjp", "fp64"])
def test_a_droplet_takes_a_few_times_a_liquid(what):
    import torch
    from paper_0709_3225_gb300 import lj
    t = []
    for x, L in (_droplet(20, 0.1, 7), inputs.jittered_fcc(20, 0.8442, 0.08, 7)):
        s = lj.System(x, None, L, precision="fp64" if what == "fp64" else "mixed", shift_mode=1)
        if what == "fp64":
            t.append(_time(lambda: lj.lj_forces(s.ctx, s.x, s.f)))
        else:
            g, dx = torch.ones_like(s.x), torch.zeros_like(s.x)
            dp = torch.zeros(2, dtype=torch.float64, device="cuda")
            t.append(_time(lambda: lj.lj_forces_vjp(s.ctx, s.x, g, 1.0, dx, dp)))
        s.check()
        s.close()
    assert t[0] <= 5.0 * t[1]


def _context_bytes(make):
    """Device memory of what make() creates beside torch's, and it."""
    import torch
    torch.cuda.synchronize()
    free, torch0 = torch.cuda.mem_get_info()[0], torch.cuda.memory_reserved()
    s = make()
    torch.cuda.synchronize()
    return free - torch.cuda.mem_get_info()[0] - (torch.cuda.memory_reserved() - torch0), s


# per particle: 32 bytes of list arrays, 4 of overflow links, and per cell 28 of counts and
# starts; 16 slots a cell where the gas alone asks for them, none where the box is too sparse
@pytest.mark.parametrize("rho,rc,slots", [(0.1, 2.5, 16), (0.8442, 1.1225, 0)])
def test_large_dilute_boxes_hold_no_wide_slots(rho, rc, slots):
    from paper_0709_3225_gb300 import lj
    n = 500000
    x, L = inputs.lattice_gas(n, rho, 3, 0.05)
    lj.System(x[:1000], None, L, rc=rc).close()   # the library's own first allocations
    held, s = _context_bytes(lambda: lj.System(x, None, L, rc=rc))
    ncell = s.ctx.nc ** 3
    s.close()
    assert held <= 36 * n + 28 * ncell + 16 * (slots * ncell + (n if slots else 0)) + (24 << 20)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_slots_widen_when_a_droplet_needs_them(oracle_mod, precision):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = _droplet(29, 0.1, 33)              # 59,319 cells: 16 slots at first
    s = lj.System(x, None, L, precision=precision, shift_mode=1)
    lj.lj_set_graph(s.ctx)
    xl, Ll = inputs.jittered_fcc(29, 0.8442, 0.08, 7)
    liquid = lj.System(xl, None, Ll, precision=precision, shift_mode=1)
    fo = oracle_mod.forces_cells(x, L, mode=1)[0]
    tol = 1e-12 if precision == "fp64" else 5e-6
    for _ in range(3):                        # beyond the slots, then with wide ones
        s.forces()
        s.check()
        assert rel_rms(s.f.double().cpu().numpy()[:, :3], fo) <= tol
    cell_of, count, _, perm = (t.cpu().numpy() for t in s.cells())
    o = oracle_mod.bin_cells(x, L, s.ctx.nc)
    assert np.array_equal(cell_of, o[0]) and np.array_equal(count, o[1]) and np.array_equal(np.sort(perm), np.arange(s.n))
    g, dx = torch.ones_like(s.x), torch.zeros_like(s.x)
    dp = torch.zeros(2, dtype=torch.float64, device="cuda")
    t = []
    for q in (s, liquid):
        q.forces()
        if precision == "fp64":
            t.append(_time(lambda: lj.lj_forces(q.ctx, q.x, q.f)))
        else:
            t.append(_time(lambda: lj.lj_forces_vjp(q.ctx, q.x, g, 1.0, dx, dp)))
    assert t[0] <= 4.0 * t[1]                 # 72 us against 45, 116 against 83; 382 and 2,207 beyond the slots
    v = np.zeros_like(x)
    s.step(9)                                 # replayed steps on the wide slots
    oracle_mod.vv(x, v, fo, L, 9, mode=1)
    assert np.abs(min_image(s.x.cpu().numpy() - x, L)).max() <= (1e-10 if precision == "fp64" else 1e-5)
    s.check()
    s.close()
    liquid.close()


def test_a_batch_widens_its_slots(oracle_mod):
    from paper_0709_3225_gb300 import lj
    states = [_droplet(17 + r % 3, 0.1, r) for r in range(4)]   # 4 x 12,167 to 17,576 cells
    xs, Ls = [x for x, _ in states], [L for _, L in states]
    b = lj.Batch(xs, [np.zeros_like(x) for x in xs], Ls)
    b.set_kernel(7)
    fo = [oracle_mod.forces_cells(x, L, mode=1)[0] for x, L in states]
    for _ in range(3):
        b.forces()
        b.check()
        for r in range(4):
            assert rel_rms(b.replica(b.f, r).double().cpu().numpy()[:, :3], fo[r]) <= 5e-6
    b.step(5)
    b.check()
    for r in range(4):
        x, v = xs[r].copy(), np.zeros_like(xs[r])
        oracle_mod.vv(x, v, fo[r], Ls[r], 5, mode=1)
        assert np.abs(min_image(b.replica(b.x, r).cpu().numpy() - x, Ls[r])).max() <= 1e-5
    b.close()


def test_a_recorded_context_keeps_its_slots(oracle_mod):
    """Slots are not widened once calls have been recorded into a caller's
    graph, which holds their addresses."""
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = _droplet(29, 0.1, 34)
    fo = oracle_mod.forces_cells(x, L, mode=1)[0]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = lj.System(x, None, L, shift_mode=1, stream=st)
        s.forces()                            # asks for wider slots
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            lj.lj_forces(s.ctx, s.x, s.f)
        for _ in range(2):
            for call in (g.replay, lambda: lj.lj_forces(s.ctx, s.x, s.f)):
                s.f.fill_(float("nan"))
                call()
                torch.cuda.synchronize()
                assert rel_rms(s.f.double().cpu().numpy()[:, :3], fo) <= 5e-6
        s.check()
        s.close()


def test_widening_leaves_another_streams_capture_alone(oracle_mod):
    import torch
    from paper_0709_3225_gb300 import lj
    x, L = _droplet(29, 0.1, 35)
    fo = oracle_mod.forces_cells(x, L, mode=1)[0]
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    s = lj.System(x, None, L, shift_mode=1, stream=st)
    torch.cuda.synchronize()
    s.forces()                                # asks for wider slots
    torch.cuda.synchronize()
    a = torch.ones(8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=other):
        a.mul_(2.0)
        s.forces()                            # not part of the capture: widens
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(a, torch.full_like(a, 2.0))
    s.forces()
    torch.cuda.synchronize()
    s.check()
    assert rel_rms(s.f.double().cpu().numpy()[:, :3], fo) <= 5e-6
    s.close()
