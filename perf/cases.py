"""The workloads whose speed is followed, over the range the library serves.

Each case is one call (or one gradient) of the public interface on a state a
program holds: a context, positions, velocities and forces on the device (or
pinned host arrays), theta, rand48 streams.  Starting configurations are FCC
sites, with random vacancies where N is no 4 m^3, every coordinate displaced
at random by as much as leaves no two particles nearer than 0.9 sigma.

``exact`` restates the calls in FP64 torch: pair lists by cells, the
truncated / shifted Lennard-Jones terms, velocity Verlet, BAOAB, the adjoint
and the rand48 series.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0709_3225_gb300 import autograd, inputs, lj

RC, DT = 2.5, 0.005
HALF = [(0, 0, 0)] + [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
                      if (dz, dy, dx) > (0, 0, 0)]


def _case(kind, name=None, **kw):
    c = {"kind": kind, "n": 0, "rho": 0.8442, "kT": 1.0, "steps": 1, "mode": 1, "precision": "mixed"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one energy evaluation of the smallest liquid workload: a call whose launches and read-back are its time
        _case("forces", "energy_2k", n=2048, kT=0.728, energy=True),
        # the smallest liquid workload stepped: five short kernels a step
        _case("step", "step_2k", n=2048, kT=0.728, steps=10),
        # the accuracy workload: the middle of the range, where the last wave of cells counts
        _case("step", "step_131k", n=131072, kT=0.728, steps=10),
        # the headline workload
        _case("step", "step_4m", n=4000000, steps=5),
        # the same physics in FP64, as a check on the mixed precision is run
        _case("step", "step_fp64_131k", n=131072, kT=0.728, steps=5, precision="fp64"),
        # the headline workload's call on host arrays, at a size a coupled host program exchanges
        _case("host", "host_500k", n=500009, steps=1),
        # a thermostatted gas of the density study, odd N, the paper's force-shifted potential
        _case("langevin", "langevin_gas_100k", n=100003, rho=0.3, steps=5, mode=2),
        # force matching: forces and the gradient of their misfit
        _case("vjp", "force_match_32k", n=32000, mode=2),
        # force matching through a trajectory, a checkpoint every 10 steps
        _case("trajectory", "trajectory_32k", n=32000, steps=10, mode=2),
        # many small replicas of uneven size, with the tuner's choice of kernel
        _case("ensemble", "ensemble_64", nrep=64, n_hi=50000, kernel=7, steps=5),
        # the paper's generator at its largest, with its number of streams
        _case("rand48", "rand48_41m", n=6144 * 6667, streams=6144, real=False),
        # the paper's first algorithm, at a size of its break-even study
        _case("all_pairs", "all_pairs_8788", n=8788, energy=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("forces", "step", "step", "host", "langevin", "vjp", "trajectory", "ensemble", "rand48",
                       "all_pairs"))
    c = _case(kind, rho=round(rng.choice((0.8442, rng.uniform(0.1, 1.0), rng.uniform(0.6, 0.9))), 4),
              kT=round(rng.uniform(0.7, 1.5), 3), mode=rng.choice((0, 1, 1, 2, 2)))
    if kind == "forces":
        c.update(n=_log(rng, 1000, 4000000), energy=rng.random() < 0.5)
    elif kind == "step":
        c.update(n=_log(rng, 1000, 4000000), steps=rng.randint(1, 5))
        if rng.random() < 0.3:
            c.update(n=_log(rng, 1000, 500000), precision="fp64")
    elif kind == "host":
        c.update(n=_log(rng, 1000, 1000000), steps=rng.randint(1, 3))
    elif kind == "langevin":
        c.update(n=_log(rng, 1000, 1000000), steps=rng.randint(1, 5))
    elif kind == "vjp":
        c.update(n=_log(rng, 1000, 500000), mode=rng.choice((1, 2)), precision=rng.choice(("mixed", "mixed", "fp64")))
    elif kind == "trajectory":
        c.update(n=_log(rng, 1000, 131072), steps=rng.randint(3, 12), mode=2)
    elif kind == "ensemble":
        c.update(nrep=rng.randint(4, 80), n_hi=rng.choice((5000, 50000)), kernel=rng.choice((3, 7, 7)),
                 steps=rng.randint(1, 5))
    elif kind == "rand48":
        streams = _log(rng, 256, 622592)
        c.update(streams=streams, n=streams * max(1, _log(rng, 10240, 40960000) // streams), real=rng.random() < 0.5)
    else:
        c.update(n=_log(rng, 1000, 32000), energy=rng.random() < 0.5)
    return c


# ---- states ------------------------------------------------------------------

def _positions(n, rho, seed):
    m = 1
    while 4 * m ** 3 < n:
        m += 1
    a = inputs.box_side(n, rho) / m
    jitter = max(0.02, (math.sqrt(0.5) - 0.9 / a) / math.sqrt(8.0))   # in lattice constants
    return inputs.lattice_gas(n, rho, seed, jitter)


def _ensemble(case, seed):
    sizes = np.random.default_rng(2024)   # the replicas' sizes and densities are the case's, the states the seed's
    n = sizes.integers(500, case["n_hi"] + 1, case["nrep"])
    rho = sizes.uniform(0.7, 0.9, case["nrep"])
    rng = np.random.default_rng(seed)
    xs, vs, boxes = [], [], []
    for r in range(case["nrep"]):
        x, L = _positions(int(n[r]), float(rho[r]), seed + 7919 * r)
        xs.append(x)
        vs.append(inputs.velocities(int(n[r]), float(rng.uniform(0.7, 1.5)), seed + 104729 * r))
        boxes.append(L)
    return xs, vs, boxes


def _fluid(case, seed):
    x, L = _positions(case["n"], case["rho"], seed)
    return x, inputs.velocities(case["n"], case["kT"], seed + 1), L


def _targets(case, seed, x):
    """Reference forces (vjp) or positions (trajectory) a fit is made to."""
    g = np.random.default_rng(seed + 2).standard_normal(x.shape)
    return 20.0 * g if case["kind"] == "vjp" else x + 0.1 * g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rand48":
        state = torch.empty(case["streams"], dtype=torch.int64, device="cuda")
        lj.lj_rand48_seed(state, lj.lj_srand48_state(seed))
        out = torch.empty(case["n"], dtype=torch.float64 if case["real"] else torch.int32, device="cuda")
        return {"case": case, "state": state, "out": out}
    if kind == "ensemble":
        batch = lj.Batch(*_ensemble(case, seed))
        batch.set_kernel(case["kernel"])
        batch.forces()
        return {"case": case, "batch": batch}
    x, v, L = _fluid(case, seed)
    s = lj.System(x, v, L, shift_mode=case["mode"], precision=case["precision"], dt=DT, rc=RC)
    s.forces()
    st = {"case": case, "system": s, "box": L}
    if kind == "langevin":
        s.langevin_seed(seed)
    if kind == "host":
        s.check()
        for k, t in (("x", s.x), ("v", s.v), ("f", s.f)):
            st[k] = torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)
    if kind in ("vjp", "trajectory"):
        st["theta"] = torch.tensor([0.9, 1.05], dtype=torch.float64, device="cuda", requires_grad=True)
        st["target"] = torch.as_tensor(_targets(case, seed, x)).cuda()
        st["x"] = s.x.clone().requires_grad_(True)
        st["v"] = s.v.clone().requires_grad_(True)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "rand48":
        fn = lj.lj_rand48_drand if case["real"] else lj.lj_rand48_lrand
        fn(st["state"], case["n"] // case["streams"], st["out"])
        return {"out": st["out"], "state": st["state"]}
    if kind == "ensemble":
        b = st["batch"]
        b.step(case["steps"])
        return {"x": b.x, "v": b.v, "f": b.f}
    s = st["system"]
    if kind == "forces":
        r = s.forces(energy=case["energy"])
        return {"f": s.f, "e": r[0], "w": r[1]} if r else {"f": s.f}
    if kind == "all_pairs":
        r = lj.lj_forces_n2(s.ctx, s.x, s.f, energy=case["energy"])
        return {"f": s.f, "e": r[0], "w": r[1]} if r else {"f": s.f}
    if kind == "step":
        s.step(case["steps"])
        return {"x": s.x, "v": s.v, "f": s.f}
    if kind == "langevin":
        s.langevin_step(case["steps"], 1.0, case["kT"])
        return {"x": s.x, "v": s.v, "f": s.f}
    if kind == "host":
        lj.lj_step_host(s.ctx, st["x"], st["v"], st["f"], case["steps"])
        return {"x": st["x"], "v": st["v"], "f": st["f"]}
    n, L = case["n"], st["box"]
    if kind == "vjp":
        F = autograd.forces(st["x"], st["theta"], s.ctx)
        loss = ((F - st["target"]) ** 2).sum() / n
        gx, gt = torch.autograd.grad(loss, (st["x"], st["theta"]))
        return {"F": F, "loss": loss, "gx": gx, "gtheta": gt}
    xT, vT = autograd.trajectory(st["x"], st["v"], st["theta"], s.ctx, case["steps"], 10)
    d = xT - st["target"]
    d = d - L * torch.round(d / L)
    loss = (d ** 2).sum() / n
    gx, gv, gt = torch.autograd.grad(loss, (st["x"], st["v"], st["theta"]))
    return {"x": xT, "v": vT, "loss": loss, "gx": gx, "gv": gv, "gtheta": gt}


# ---- what a pass cannot do without ---------------------------------------------

def _pairs_in_range(n, rho):
    return n * (2.0 / 3.0) * math.pi * RC ** 3 * rho


def work(case):
    """20 operations a pair within rc (40 for its adjoint term), as the force
    is counted elsewhere; each input read once, each output written once."""
    kind, n, k = case["kind"], case["n"], case["steps"]
    fb = 32 if case["precision"] == "fp64" else 16
    if kind == "rand48":
        return {"bytes": n * (8 if case["real"] else 4) + 16 * case["streams"], "flops": 0}
    if kind == "ensemble":
        n = case["nrep"] * (500 + case["n_hi"]) // 2
        return {"bytes": n * 2 * (48 + fb), "flops": 20.0 * k * _pairs_in_range(n, 0.8)}
    p = _pairs_in_range(n, case["rho"])
    if kind == "forces":
        return {"bytes": n * (24 + fb), "flops": 20.0 * p}
    if kind == "all_pairs":
        return {"bytes": n * (24 + fb), "flops": 12.0 * n * (n - 1.0) / 2.0}
    if kind in ("step", "host"):
        return {"bytes": n * 2 * (48 + fb), "flops": 20.0 * k * p}
    if kind == "langevin":
        return {"bytes": n * 2 * (48 + fb + 8), "flops": 20.0 * k * p}
    if kind == "vjp":
        return {"bytes": n * 24 * 4, "flops": 60.0 * p}
    return {"bytes": n * 24 * 7, "flops": (20.0 + 20.0 + 80.0) * k * p}


# ---- the same in FP64, by plain torch --------------------------------------------

def _pairs(x, L):
    """Indices (i, j) of the pairs within RC at the minimum image, each once."""
    n, dev = x.shape[0], x.device
    nc = int(L / RC)
    w = x - L * torch.floor(x / L)
    c = (w * (nc / L)).long().clamp_(0, nc - 1)
    cid = c[:, 0] + nc * (c[:, 1] + nc * c[:, 2])
    order = torch.argsort(cid)
    count = torch.bincount(cid, minlength=nc ** 3)
    start = torch.cumsum(count, 0) - count
    occ = int(count.max())
    table = torch.full((nc ** 3, occ), n, dtype=torch.int64, device=dev)
    table[cid[order], torch.arange(n, device=dev) - start[cid[order]]] = order
    xp = torch.cat([w, torch.full((1, 3), float("nan"), dtype=w.dtype, device=dev)])
    ids = torch.arange(nc ** 3, device=dev)
    cx, cy, cz = ids % nc, (ids // nc) % nc, ids // (nc * nc)
    upper = torch.ones(occ, occ, dtype=torch.bool, device=dev).triu(1)
    chunk = max(1, 20_000_000 // (occ * occ))
    ii, jj = [], []
    for dx, dy, dz in HALF:
        nb = (cx + dx) % nc + nc * ((cy + dy) % nc + nc * ((cz + dz) % nc))
        for c0 in range(0, nc ** 3, chunk):
            a, b = table[c0:c0 + chunk], table[nb[c0:c0 + chunk]]
            d = xp[a][:, :, None, :] - xp[b][:, None, :, :]
            d -= L * torch.round(d / L)
            keep = (d * d).sum(-1) < RC * RC     # false for the empty slots (NaN)
            if (dx, dy, dz) == (0, 0, 0):
                keep &= upper
            q, s, t = keep.nonzero(as_tuple=True)
            ii.append(a[q, s])
            jj.append(b[q, t])
    return torch.cat(ii), torch.cat(jj)


def _terms(x, L, eps, sigma, mode):
    """The pairs, their d = x_i - x_j, r^2, F(r)/r and U(r)."""
    i, j = _pairs(x, L)
    d = x[i] - x[j]
    d -= L * torch.round(d / L)
    r2 = (d * d).sum(-1)
    s6 = sigma ** 6 / r2 ** 3
    phi = 24.0 * eps * (2.0 * s6 * s6 - s6) / r2
    u = 4.0 * eps * (s6 * s6 - s6)
    c6 = sigma ** 6 / RC ** 6
    fc = 24.0 * eps * (2.0 * c6 * c6 - c6) / RC
    if mode >= 1:
        u = u - 4.0 * eps * (c6 * c6 - c6)
    if mode == 2:
        r = torch.sqrt(r2)
        phi = phi - fc / r
        u = u + (r - RC) * fc
    return i, j, d, r2, phi, u


def _forces(x, L, mode, eps=1.0, sigma=1.0, energy=False):
    i, j, d, r2, phi, u = _terms(x, L, eps, sigma, mode)
    f = torch.zeros((x.shape[0], 4), dtype=torch.float64, device=x.device)
    fd = phi[:, None] * d
    f[:, :3].index_add_(0, i, fd)
    f[:, :3].index_add_(0, j, -fd)
    if not energy:
        return f
    f[:, 3].index_add_(0, i, 0.5 * u)
    f[:, 3].index_add_(0, j, 0.5 * u)
    return f, u.sum().item(), (phi * r2).sum().item()


def _vjp(x, g, L, mode, eps, sigma):
    """(dL/dx, dL/d(eps, sigma)) for dL/dF = g, rc held fixed."""
    i, j, d, r2, phi, _ = _terms(x, L, eps, sigma, mode)
    s6 = sigma ** 6 / r2 ** 3
    dphi = 24.0 * eps * (8.0 * s6 - 28.0 * s6 * s6) / (r2 * r2)     # phi'(r) / r
    dsig = 24.0 * eps * (24.0 * s6 * s6 - 6.0 * s6) / (r2 * sigma)
    if mode == 2:
        r = torch.sqrt(r2)
        c6 = sigma ** 6 / RC ** 6
        dphi = dphi + 24.0 * eps * (2.0 * c6 * c6 - c6) / RC / (r * r2)
        dsig = dsig - 24.0 * eps * (24.0 * c6 * c6 - 6.0 * c6) / (RC * sigma) / r
    h = g[i] - g[j]
    dot = (d * h).sum(-1)
    t = phi[:, None] * h + (dphi * dot)[:, None] * d
    dx = torch.zeros_like(x)
    dx.index_add_(0, i, t)
    dx.index_add_(0, j, -t)
    return dx, torch.stack([(phi * dot).sum() / eps, (dsig * dot).sum()])


def _verlet(x, v, L, mode, steps, eps=1.0, sigma=1.0):
    """Velocity Verlet: the positions of every step, the last v and f."""
    f = _forces(x, L, mode, eps, sigma)
    states = [x]
    for _ in range(steps):
        v = v + 0.5 * DT * f[:, :3]
        x = x + DT * v
        x = x - L * torch.floor(x / L)
        f = _forces(x, L, mode, eps, sigma)
        v = v + 0.5 * DT * f[:, :3]
        states.append(x)
    return states, v, f


MASK = (1 << 48) - 1


def _jump(m):
    """(A, C) of m steps of x -> a x + c mod 2^48."""
    A, C, pa, pc = 1, 0, 0x5DEECE66D, 0xB
    while m:
        if m & 1:
            A, C = pa * A & MASK, pa * C + pc & MASK
        pa, pc, m = pa * pa & MASK, pa * pc + pc & MASK, m >> 1
    return A, C


def _series(x0, m, dev):
    """x_1 .. x_m of the rand48 series from x0, by doubling."""
    A, C = _jump(1)
    s = torch.tensor([A * x0 + C & MASK], dtype=torch.int64, device=dev)
    while s.numel() < m:
        A, C = _jump(s.numel())
        s = torch.cat([s, (s * A + C) & MASK])   # int64 products wrap mod 2^64
    return s[:m]


def _normals(a, b):
    r = torch.sqrt(-2.0 * torch.log(1.0 - a.double() * 2.0 ** -48))
    t = 2.0 * math.pi * (b.double() * 2.0 ** -48)
    return r * torch.cos(t), r * torch.sin(t)


def _langevin(x, v, L, mode, steps, kT, seed, gamma=1.0):
    n = x.shape[0]
    u = _series((seed & 0xFFFFFFFF) << 16 | 0x330E, 4 * steps * n, x.device).reshape(steps, 4, n)
    c1 = math.exp(-gamma * DT)
    c2 = math.sqrt(1.0 - c1 * c1) * math.sqrt(kT)
    f = _forces(x, L, mode)
    for s in range(steps):
        z0, z1 = _normals(u[s, 0], u[s, 1])
        z2, _ = _normals(u[s, 2], u[s, 3])
        v = v + 0.5 * DT * f[:, :3]
        x = x + 0.5 * DT * v
        v = c1 * v + c2 * torch.stack([z0, z1, z2], 1)
        x = x + 0.5 * DT * v
        x = x - L * torch.floor(x / L)
        f = _forces(x, L, mode)
        v = v + 0.5 * DT * f[:, :3]
    return x, v, f


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind, mode, k = case["kind"], case["mode"], case["steps"]
    if kind == "rand48":
        s = _series((seed & 0xFFFFFFFF) << 16 | 0x330E, case["n"] + case["streams"], dev)
        out = s[:case["n"]]
        return {"out": out.double() * 2.0 ** -48 if case["real"] else (out >> 17).int(), "state": s[case["n"]:]}
    if kind == "ensemble":
        got = []
        for x, v, L in zip(*_ensemble(case, seed)):
            states, v, f = _verlet(torch.as_tensor(x, device=dev), torch.as_tensor(v, device=dev), L, mode, k)
            got.append((states[-1], v, f))
        x, v, f = (torch.cat(t) for t in zip(*got))
        return {"x": x, "v": v, "f": f}
    x, v, L = _fluid(case, seed)
    target = torch.as_tensor(_targets(case, seed, x), device=dev)
    x, v = torch.as_tensor(x, device=dev), torch.as_tensor(v, device=dev)
    n = case["n"]
    if kind in ("forces", "all_pairs"):
        if not case["energy"]:
            return {"f": _forces(x, L, mode)}
        f, e, w = _forces(x, L, mode, energy=True)
        return {"f": f, "e": e, "w": w}
    if kind in ("step", "host"):
        states, v, f = _verlet(x, v, L, mode, k)
        return {"x": states[-1], "v": v, "f": f}
    if kind == "langevin":
        x, v, f = _langevin(x, v, L, mode, k, case["kT"], seed)
        return {"x": x, "v": v, "f": f}
    eps, sigma = 0.9, 1.05
    if kind == "vjp":
        F = _forces(x, L, mode, eps, sigma)[:, :3]
        gx, gt = _vjp(x, 2.0 / n * (F - target), L, mode, eps, sigma)
        return {"F": F, "loss": ((F - target) ** 2).sum() / n, "gx": gx, "gtheta": gt}
    states, vT, _ = _verlet(x, v, L, mode, k, eps, sigma)
    d = states[-1] - target
    d = d - L * torch.round(d / L)
    lx, lv, gt = 2.0 / n * d, torch.zeros_like(d), torch.zeros(2, dtype=torch.float64, device=dev)
    for s in range(k - 1, -1, -1):
        gx, gp = _vjp(states[s + 1], 0.5 * DT * lv, L, mode, eps, sigma)
        lx, gt = lx + gx, gt + gp
        lv = lv + DT * lx
        gx, gp = _vjp(states[s], 0.5 * DT * lv, L, mode, eps, sigma)
        lx, gt = lx + gx, gt + gp
    return {"x": states[-1], "v": vT, "loss": (d ** 2).sum() / n, "gx": lx, "gv": lv, "gtheta": gt}
