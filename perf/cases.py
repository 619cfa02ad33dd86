"""Performance cases: the time stepping a user of this package runs, from a coarse tank to the largest one.

A case is a dict of plain values.  ``prepare`` builds the simulation (or the MPS tank) and loads a seeded state, ``run``
advances it through the package's entry points, ``exact`` advances the same state in plain FP64 PyTorch, ``work`` counts
what the path cannot do without.

The state a simulation advances lives in the workspace tensor its owner allocated (``Simulation.workspace``,
``mps.Tank.workspace``): its first arrays are, in particle-id order, the positions (x, y, z, 0), then the velocities with
the density (mixed form: the FP32 offset rho - rho0), then the previous level; the MPS tank holds positions, velocities,
and further on the pressures.  ``run`` returns them in place, so a pass is the stepping and nothing else; only the
monitored case also reads probes back, as a program that records gauges does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_01959_gb300 import mps, sph, workloads as wl

G = 9.81
RHO0 = 1000.0
LAYERS = 2
FLUID, BOUNDARY, GATE = 0, 1, 3


def listed():
    base = dict(path="wcsph", form="mixed", integrator="verlet", params="standard", delta="all", instances=1,
                once=False, probes=False)
    return [
        # the smallest calls: the coarse dam break a user develops and tests with (18,532 particles), both forms
        dict(base, name="small_fp64", shape="small", dp=0.02, form="fp64", steps=16),
        dict(base, name="small_mixed", shape="small", dp=0.02, steps=16),
        # a monitored run: one step, then the gauges (pressures, wave heights, force) are read; ragged spacing
        dict(base, name="monitored_step", shape="obstacle", dp=0.0171, form="fp64", steps=1, probes=True),
        # the ordinary run: obstacle dam break, 0.9 M particles, mixed and FP64
        dict(base, name="obstacle_mixed", shape="obstacle", dp=0.01, steps=16),
        dict(base, name="obstacle_fp64", shape="obstacle", dp=0.01, form="fp64", steps=2),
        # FP64 with the other options in use: symplectic scheme, delta term over full supports, ragged spacing
        dict(base, name="fp64_symplectic", shape="obstacle", dp=0.0193, form="fp64", integrator="symplectic",
             delta="full", steps=2),
        # the paper's own smoothing length and sound speed at its Case 1 resolution (2.0 M particles)
        dict(base, name="paper_mixed", shape="obstacle", dp=0.0075, params="paper", steps=16),
        # moving gate under the predictor-corrector (1.07 M particles, two pair passes per step)
        dict(base, name="gate_symplectic", shape="gate", dp=0.005, integrator="symplectic", steps=16),
        # a batch of 64 dam breaks advanced together (alpha sweep, 2.8 M particles)
        dict(base, name="sweep_mixed", shape="sweep", dp=0.0, instances=64, steps=16),
        # the largest single tank (8.1 M particles)
        dict(base, name="wall_impact_mixed", shape="wall", dp=0.0025, steps=16),
        # the MPS step: a coarse tank (many small launches) and the Case 1 tank (2.2 M particles)
        dict(name="mps_coarse", path="mps", tank_x=1.0, tank_y=0.5, tank_z=0.5, col_x=0.4, col_y=0.5, col_z=0.3,
             dp=0.02, steps=1),
        dict(name="mps_case1", path="mps", tank_x=3.22, tank_y=1.0, tank_z=1.0, col_x=1.2, col_y=1.0, col_z=0.55,
             dp=0.0075, steps=1),
    ]


# spacings each shape is run at: from a few thousand particles to the listed ones' size
RANGES = {"small": (0.008, 0.03), "obstacle": (0.0095, 0.04), "wall": (0.006, 0.03), "gate": (0.006, 0.02)}


def draw(rng):
    def spread(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    if rng.random() < 0.2:
        return dict(path="mps", tank_x=round(rng.uniform(0.9, 3.2), 3), tank_y=round(rng.uniform(0.3, 1.0), 3),
                    tank_z=round(rng.uniform(0.5, 1.0), 3), col_x=round(rng.uniform(0.3, 0.8), 3), col_y=0.3,
                    col_z=round(rng.uniform(0.2, 0.45), 3), dp=round(spread(0.0125, 0.035), 5),
                    steps=rng.choice([1, 2, 3]))
    form = "fp64" if rng.random() < 0.3 else "mixed"
    case = dict(path="wcsph", form=form, integrator="symplectic" if rng.random() < 0.25 else "verlet",
                params="paper" if rng.random() < 0.25 else "standard", delta="full" if rng.random() < 0.25 else "all",
                instances=1, once=form == "fp64" and rng.random() < 0.25, probes=form == "fp64" and rng.random() < 0.35)
    if case["once"]:
        case["delta"] = "all"
    if rng.random() < 0.2:
        case.update(shape="sweep", dp=0.0, instances=rng.randint(2, 40 if form == "mixed" else 8),
                    params="standard", probes=False)
    else:
        shape = rng.choice(sorted(RANGES))
        lo, hi = RANGES[shape]
        case.update(shape=shape, dp=round(spread(lo * (2.0 if form == "fp64" else 1.0), hi), 5))
    case["steps"] = rng.choice([1, 2, 4]) if form == "fp64" else rng.choice([1, 7, 16, 23])
    return case


# --------------------------------------------------------------------------- inputs
def _tanks(case, seed):
    """The workloads.Case of every instance."""
    shape, dp = case["shape"], case["dp"]
    if shape == "sweep":
        return wl.alpha_sweep(case["instances"], seed=2306)
    if shape == "small":
        c = wl.Case("small", (1.0, 0.5, 0.5), (0.4, 0.5, 0.3), None, dp)
    elif shape == "obstacle":
        c = wl.Case("obstacle", (3.2, 1.0, 1.0), (1.2, 1.0, 0.55), (2.4, 0.3, 0.0, 0.16, 0.4, 0.16), dp)
    elif shape == "wall":
        c = wl.Case("wall", (1.6, 0.6, 0.6), (0.6, 0.6, 0.3), None, dp)
    else:
        c = wl.gate_dambreak(dp)
    return [wl.paper_parameters(c) if case["params"] == "paper" else c]


def _nint(x):
    return int(math.floor(x + 0.5))


def _box(i0, j0, k0, nx, ny, nz):
    k, j, i = np.meshgrid(np.arange(k0, k0 + nz), np.arange(j0, j0 + ny), np.arange(i0, i0 + nx), indexing="ij")
    return np.stack([i.ravel(), j.ravel(), k.ravel()], 1)


def _shell(tank, dp, layers):
    nt = [_nint(v / dp) for v in tank]
    b = _box(-layers, -layers, -layers, nt[0] + 2 * layers, nt[1] + 2 * layers, nt[2] + layers)
    inside = (b[:, 0] >= 0) & (b[:, 0] < nt[0]) & (b[:, 1] >= 0) & (b[:, 1] < nt[1]) & (b[:, 2] >= 0)
    return b[~inside], nt


def _lattice(c):
    """Positions and types of one tank in particle-id order: fluid, walls and floor, obstacle, gate."""
    dp = c.dp
    parts = [_box(0, 0, 0, *[_nint(v / dp) for v in c.column]), _shell(c.tank, dp, LAYERS)[0]]
    kinds = [FLUID, BOUNDARY]
    for box, kind in ((c.obstacle, BOUNDARY), (c.gate, GATE)):
        if box is not None:
            parts.append(_box(*[_nint(v / dp) for v in box]))
            kinds.append(kind)
    r = (np.concatenate(parts) + 0.5) * dp
    return r, np.repeat(np.array(kinds, np.int32), [len(p) for p in parts])


def _noise(rng, n):
    return rng.random((n, 3), dtype=np.float32) - np.float32(0.5)


def _wcsph_inputs(case, seed):
    """Every instance's (case, r, u, rho, type): the collapsing column, its lattice disturbed by a tenth of a spacing, a
    smooth seeded velocity field with small noise, hydrostatic densities with small noise.  Velocities and density
    offsets are FP32 values, so that both forms hold them exactly."""
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for c in _tanks(case, seed):
        r, kind = _lattice(c)
        n, nf = len(r), int(np.count_nonzero(kind == FLUID))
        r[:nf] += (0.2 * c.dp) * _noise(rng, nf)
        u = np.zeros((n, 3), np.float32)
        amp, phase = rng.uniform(0.2, 0.6, 3), rng.uniform(0.0, 2.0 * math.pi, 3)
        lx, ly, lz = c.column
        x, y, z = r[:nf, 0] / lx, r[:nf, 1] / ly, r[:nf, 2] / lz
        u[:nf, 0] = amp[0] * x * (1.2 - z) + 0.1 * np.sin(3.0 * y + phase[0])
        u[:nf, 1] = 0.1 * np.sin(3.0 * x + phase[1]) * y * (1.0 - y)
        u[:nf, 2] = -amp[2] * z * x + 0.02 * np.sin(3.0 * y + phase[2])
        u[:nf] += np.float32(0.04) * _noise(rng, nf)
        u[kind == GATE] = np.asarray(c.gate_velocity, np.float32)
        d = np.zeros(n, np.float32)
        hc = c.column[2]
        d[:nf] = RHO0 * ((1.0 + 7.0 * G * np.maximum(hc - r[:nf, 2], 0.0) / c.c0**2) ** (1.0 / 7.0) - 1.0)
        d += np.float32(0.1) * (rng.random(n, dtype=np.float32) - np.float32(0.5))
        out.append((c, r, u.astype(np.float64), RHO0 + d.astype(np.float64), kind))
    return out


def _mps_inputs(case, seed):
    """Positions, velocities, types (0 fluid, 1 wall, 2 dummy), spacing and time step of an MPS tank."""
    rng = np.random.Generator(np.random.PCG64(seed))
    dp = case["dp"]
    tank = (case["tank_x"], case["tank_y"], case["tank_z"])
    col = (case["col_x"], case["col_y"], case["col_z"])
    fluid = _box(0, 0, 0, *[_nint(v / dp) for v in col])
    shell, nt = _shell(tank, dp, 3)
    low = np.maximum(-1 - shell, -1)
    high = np.maximum(shell - np.asarray(nt), -1)
    high[:, 2] = -1
    layer = np.maximum(low, high).max(1)
    nf = len(fluid)
    r = (np.concatenate([fluid, shell]) + 0.5) * dp
    kind = np.concatenate([np.zeros(nf, np.int32), np.where(layer == 0, 1, 2).astype(np.int32)])
    u = np.zeros_like(r)
    r[:nf] += 0.05 * dp * _noise(rng, nf)
    amp = rng.uniform(0.1, 0.3)
    u[:nf, 0] = amp * r[:nf, 0] / col[0] * (1.2 - r[:nf, 2] / col[2])
    u[:nf, 2] = -amp * r[:nf, 2] / col[2] * r[:nf, 0] / col[0]
    u[:nf] += 0.01 * _noise(rng, nf)
    return tank, col, r, u, kind, 3.0e-4 * dp / 0.0075


def prepare(case, seed):
    if case["path"] == "mps":
        tank, col, r, u, kind, dt = _mps_inputs(case, seed)
        t = mps.Tank(tank, col, case["dp"], dt)
        t.set_state(r, u)
        return dict(case=case, tank=t)
    parts = _wcsph_inputs(case, seed)
    kw = dict(precision=sph.FP64 if case["form"] == "fp64" else sph.MIXED,
              integrator=sph.SYMPLECTIC if case["integrator"] == "symplectic" else sph.VERLET,
              delta_mode=sph.DELTA_FULL_SUPPORT if case["delta"] == "full" else sph.DELTA_ALL_FLUID,
              pair_symmetric=1 if case["once"] else 0)
    sim = sph.Simulation([p[0] for p in parts], batch=len(parts) > 1, **kw)
    sim.set_state(*[np.concatenate([p[k] for p in parts]) if len(parts) > 1 else parts[0][k] for k in (1, 2, 3)])
    return dict(case=case, sim=sim)


# --------------------------------------------------------------------------- one pass
def _array(workspace, offset, n, width, dtype):
    """(array of n x width values at `offset`, the 256-byte aligned offset after it)."""
    size = n * width * torch.empty(0, dtype=dtype).element_size()
    a = workspace[offset:offset + size].view(dtype)
    return (a.view(n, width) if width > 1 else a), (offset + size + 255) // 256 * 256


def run(state):
    case = state["case"]
    if case["path"] == "mps":
        t = state["tank"]
        t.step(case["steps"])
        pos, o = _array(t.workspace, 0, t.n, 4, torch.float64)
        vel, o = _array(t.workspace, o, t.n, 4, torch.float64)
        _, o = _array(t.workspace, o, t.n, 4, torch.float64)
        for _ in range(2):
            _, o = _array(t.workspace, o, t.n, 1, torch.uint8)
        return dict(position=pos, velocity=vel, pressure=_array(t.workspace, o, t.n, 1, torch.float64)[0])
    sim = state["sim"]
    sim.step(0.0, case["steps"])
    vt = torch.float64 if case["form"] == "fp64" else torch.float32
    pos, o = _array(sim.workspace, 0, sim.n, 4, torch.float64)
    vel, o = _array(sim.workspace, o, sim.n, 4, vt)
    out = dict(position=pos, velocity=vel, previous=_array(sim.workspace, o, sim.n, 4, vt)[0])
    if case["probes"]:
        c = sim.cases[0]
        pts, xy = _gauges(c)
        out["pressure"] = sim.probe_pressure(pts)
        out["height"] = sim.probe_wave_height(xy)
        if c.obstacle is not None:
            out["force"] = sim.probe_force()
    return out


def _gauges(c):
    lx, ly, lz = c.column
    x, z = np.meshgrid(np.linspace(0.1, 0.9, 4) * lx, np.linspace(0.1, 0.7, 3) * lz)
    pts = np.stack([x.ravel(), np.full(x.size, 0.47 * ly), z.ravel()], 1)
    xy = np.stack([np.linspace(0.05, 0.85, 4) * lx, np.full(4, 0.53 * ly)], 1)
    return pts, xy


# --------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["path"] == "mps":
        dp = case["dp"]
        nf = _nint(case["col_x"] / dp) * _nint(case["col_y"] / dp) * _nint(case["col_z"] / dp)
        nt = [_nint(case[k] / dp) for k in ("tank_x", "tank_y", "tank_z")]
        n = nf + (nt[0] + 6) * (nt[1] + 6) * (nt[2] + 3) - nt[0] * nt[1] * nt[2]
        # state once in and out, and per iteration (about 20 + 0.9 per layer of the column's depth, from runs) the
        # off-diagonal matrix entries (value and column) and six vectors
        its = 20 + 0.9 * (case["col_z"] + case["col_x"]) / dp / 2
        return dict(bytes=case["steps"] * (n * 136 + its * nf * (32 * 12 + 48)),
                    flops=case["steps"] * (nf * 32 * 90 + its * nf * (2 * 33 + 12)))
    n = pairs = 0
    for c in _tanks(case, 0):
        nf, nw, no = c.lattice_counts(LAYERS)
        near = 4.0 / 3.0 * math.pi * (2.0 * c.h / c.dp) ** 3
        n += nf + nw + no
        pairs += nf * near + 0.2 * (nw + no) * near
    passes = case["steps"] * (2 if case["integrator"] == "symplectic" else 1)
    per = 32 + 64 if case["form"] == "fp64" else 32 + 32
    # per step the state in and out; 80 floating-point operations per interacting ordered pair
    return dict(bytes=case["steps"] * n * 2 * per, flops=passes * pairs * 80)


# --------------------------------------------------------------------------- the same in plain FP64 PyTorch
MAX_EXACT = 7.0e10  # candidate pairs over all passes: about 15 s


def _neighbours(r, radius, budget=24_000_000):
    """Chunks (i, j, rij = r_i - r_j, |rij|^2) over all ordered pairs within `radius`."""
    lo = r.min(0).values - 1.5 * radius
    cell = ((r - lo) / radius).floor().long()
    dims = (cell.max(0).values + 2).tolist()
    key = (cell[:, 2] * dims[1] + cell[:, 1]) * dims[0] + cell[:, 0]
    key, order = key.sort()
    start = torch.searchsorted(key, torch.arange(dims[0] * dims[1] * dims[2] + 1, device=r.device))
    rs = r[order]
    n = len(r)
    rows = torch.tensor([(dz * dims[1] + dy) * dims[0] for dz in (-1, 0, 1) for dy in (-1, 0, 1)], device=r.device)
    at = key[:, None] + rows[None, :]
    first, count = start[at - 1], start[at + 2] - start[at - 1]
    total = count.sum(1).cumsum(0)
    i0 = 0
    while i0 < n:
        done = int(total[i0 - 1]) if i0 else 0
        i1 = max(i0 + 1, int(torch.searchsorted(total, done + budget)))
        f, k = first[i0:i1].reshape(-1), count[i0:i1].reshape(-1)
        owner = torch.repeat_interleave(torch.arange(len(k), device=r.device), k)
        j = torch.arange(len(owner), device=r.device) - (k.cumsum(0) - k - f)[owner]
        i = i0 + owner // 9
        d = rs[i] - rs[j]
        r2 = (d * d).sum(1)
        near = (r2 < radius * radius) & (i != j)
        i, j = i[near], j[near]
        yield order[i], order[j], d[near], r2[near]
        i0 = i1


def _derivatives(c, r, u, rho, kind, full):
    h, m = c.h, RHO0 * c.dp**3
    b = RHO0 * c.c0**2 / 7.0
    pr = b * ((rho / RHO0) ** 7 - 1.0)
    cs = c.c0 * (rho / RHO0) ** 3
    kf = 105.0 / (16.0 * math.pi * h**5)
    n = len(r)
    drho, dif, acc = torch.zeros_like(rho), torch.zeros_like(rho), torch.zeros_like(r)
    mumax, wall = torch.zeros_like(rho), torch.zeros_like(rho)
    fluid = kind == FLUID
    for i, j, d, r2 in _neighbours(r, 2.0 * h):
        fi, fj = fluid[i], fluid[j]
        wall.index_add_(0, i, (~fj).double())
        both = fi | fj
        i, j, d, r2, ff = i[both], j[both], d[both], r2[both], (fi & fj)[both]
        f = -kf * (1.0 - 0.5 * r2.sqrt() / h) ** 3
        ud = ((u[i] - u[j]) * d).sum(1)
        ri, rj = rho[i], rho[j]
        mu = h * ud / (r2 + 0.01 * h * h)
        visc = torch.where(ud < 0, -c.alpha * (cs[i] + cs[j]) * mu / (ri + rj), torch.zeros_like(mu))
        drho.index_add_(0, i, m * f * ud)
        dif.index_add_(0, i, torch.where(ff, -m * f * (2.0 * 0.1 * h * c.c0) * (rj - ri) / rj, torch.zeros_like(f)))
        acc.index_add_(0, i, (-m * f * ((pr[i] + pr[j]) / (ri * rj) + visc))[:, None] * d)
        mumax.index_reduce_(0, i, mu, "amax")
    drho = drho + (torch.where(wall > 0, torch.zeros_like(dif), dif) if full else dif)
    acc[fluid, 2] -= G
    a = acc[fluid].square().sum(1).sqrt().max()
    dt = 0.2 * torch.minimum(torch.sqrt(h / a), h / (c.c0 + mumax[fluid].max()))
    return drho, acc, dt


def _advance(case, c, r, u, rho, kind):
    dev = torch.device("cuda")
    r, u, rho = (torch.from_numpy(np.array(a, np.float64)).to(dev) for a in (r, u, rho))
    kind = torch.from_numpy(kind).to(dev)
    fl, full = (kind == FLUID)[:, None], case["delta"] == "full"
    gv = torch.where((kind == GATE)[:, None], torch.tensor(c.gate_velocity, dtype=torch.float64, device=dev),
                     torch.zeros((), dtype=torch.float64, device=dev))
    up, rp = u.clone(), rho.clone()
    for step in range(case["steps"]):
        drho, acc, dt = _derivatives(c, r, u, rho, kind, full)
        if case["integrator"] == "symplectic":
            un, rn = u, rho
            r = r + 0.5 * dt * torch.where(fl, u, gv)
            u = torch.where(fl, u + 0.5 * dt * acc, gv)
            rho = rho + 0.5 * dt * drho
            drho, acc, _ = _derivatives(c, r, u, rho, kind, full)
            e = -dt * drho / rho
            u = torch.where(fl, un + dt * acc, gv)
            r = r + 0.5 * dt * u
            rho = rn * (2.0 - e) / (2.0 + e)
            up, rp = un, rn
        else:
            first = step % 40 == 0
            u2 = u + dt * acc if first else up + 2.0 * dt * acc
            rho2 = rho + dt * drho if first else rp + 2.0 * dt * drho
            r = torch.where(fl, r + dt * u + 0.5 * dt * dt * acc, r + dt * gv)
            up, rp = torch.where(fl, u, gv), rho
            u, rho = torch.where(fl, u2, gv), rho2
    return r, u, rho, up, rp


def _exact_mps(case, seed):
    dev = torch.device("cuda")
    tank, col, r, u, kind, dt = _mps_inputs(case, seed)
    l0, nu, rho, kc, kr, tol = case["dp"], 1e-6, 1000.0, 1e-8, 0.01, 1e-6
    re = 2.1 * l0
    r, u, kind = (torch.from_numpy(a).to(dev) for a in (r, u, kind))
    fluid, n = (kind == 0), len(r)
    k = np.arange(-3, 4)
    d = np.sqrt((np.stack(np.meshgrid(k, k, k), -1).reshape(-1, 3) ** 2).sum(1)) * l0
    d = d[d > 0]
    w = np.where(d > re, 0.0, re / d - 1.0)
    n0 = float(w.sum())
    lapc = 6.0 / (float((d * d * w).sum() / w.sum()) * n0)
    press = torch.zeros(n, dtype=torch.float64, device=dev)
    for _ in range(case["steps"]):
        lap = torch.zeros_like(u)
        for i, j, d, r2 in _neighbours(r, re):
            f = fluid[i]
            i, j, r2 = i[f], j[f], r2[f]
            lap.index_add_(0, i, (u[j] - u[i]) * (re / r2.sqrt() - 1.0)[:, None])
        g = torch.tensor([0.0, 0.0, -G], dtype=torch.float64, device=dev)
        us = torch.where(fluid[:, None], u + dt * (nu * lapc * lap + g), u)
        rs = r + dt * torch.where(fluid[:, None], us, torch.zeros_like(us))
        parts = [(i, j, -d, r2) for i, j, d, r2 in _neighbours(rs, re)]
        i, j, d, r2 = (torch.cat([p[q] for p in parts]) for q in range(4))
        w = re / r2.sqrt() - 1.0
        zero = torch.zeros(n, dtype=torch.float64, device=dev)
        nd = zero.index_add(0, i, w)
        mean = torch.zeros_like(r).index_add(0, i, d * w[:, None])
        sig = torch.where(nd > 0, mean.square().sum(1).sqrt() / nd, zero)
        surf = (kind != 2) & (nd < 0.98 * n0) & (sig > 0.2 * l0)
        unknown = (kind != 2) & ~surf
        solid = unknown[i] & (kind[j] != 2)
        diag = torch.where(unknown, lapc * zero.index_add(0, i[solid], w[solid]) + rho * kc / dt**2, zero + 1.0)
        rhs = torch.where(unknown, kr * rho / dt**2 * (nd - n0) / n0, zero)
        off = solid & unknown[j]
        a = torch.sparse_coo_tensor(torch.stack([i[off], j[off]]), -lapc * w[off], (n, n)).to_sparse_csr()
        x, res = zero.clone(), rhs.clone()
        p, rr, bb = res.clone(), float(rhs @ rhs), float(rhs @ rhs)
        while rr > 0:
            q = diag * p + a @ p
            alpha = rr / float(p @ q)
            x, res = x + alpha * p, res - alpha * q
            new = float(res @ res)
            if math.sqrt(new) <= tol * math.sqrt(bb):
                break
            p, rr = res + (new / rr) * p, new
        press = torch.where(unknown, x.clamp(min=0.0), zero)
        near = fluid[i] & (kind[j] != 2)
        i, j, d, r2, w = i[near], j[near], d[near], r2[near], w[near]
        low = press.clone().index_reduce(0, i, press[j], "amin")
        e = d / r2.sqrt()[:, None]
        mom = torch.zeros((n, 9), dtype=torch.float64, device=dev)
        mom.index_add_(0, i, (e[:, :, None] * e[:, None, :] * w[:, None, None]).reshape(-1, 9))
        v = torch.zeros_like(r).index_add(0, i, ((press[j] - low[i]) * w / r2)[:, None] * d)
        mom = mom.reshape(-1, 3, 3)
        scale = mom.diagonal(dim1=1, dim2=2).sum(1) / 3.0
        good = fluid & (torch.linalg.det(mom).abs() > 1e-12 * scale**3)
        grad = torch.zeros_like(r)
        grad[good] = torch.linalg.solve(mom[good], v[good][:, :, None])[:, :, 0]
        u = torch.where(fluid[:, None], us - dt / rho * grad, u)
        r = torch.where(fluid[:, None], rs + dt * (u - us), r)
    pad = torch.zeros((n, 1), dtype=torch.float64, device=dev)
    return dict(position=torch.cat([r, pad], 1), velocity=torch.cat([u, pad], 1), pressure=press)


def _probe_values(c, r, u, rho, kind):
    """Gauge pressures, wave heights and the obstacle force of a state, by sums over all fluid particles near each."""
    pts, xy = _gauges(c)
    h, m = c.h, RHO0 * c.dp**3
    fl = kind == FLUID
    rf, rhof = r[fl], rho[fl]
    pf = RHO0 * c.c0**2 / 7.0 * ((rhof / RHO0) ** 7 - 1.0)

    def weights(p):
        q = (rf - p).square().sum(1).sqrt() / h
        w = 21.0 / (16.0 * math.pi * h**3) * (1.0 - 0.5 * q) ** 4 * (2.0 * q + 1.0)
        return torch.where(q < 2.0, w, torch.zeros_like(w))

    dev = r.device
    pressure = []
    for p in pts:
        w = weights(torch.tensor(p, dtype=torch.float64, device=dev))
        pressure.append(float((w * pf).sum() / w.sum()) if float(w.sum()) > 0 else 0.0)
    height = []
    dz = 0.25 * c.dp
    for p in xy:
        z, level = 0.0, 0
        near = (rf[:, 0] - p[0]) ** 2 + (rf[:, 1] - p[1]) ** 2 < 4.0 * h * h
        rn = rf[near]
        zs = torch.arange(int((c.tank[2] + 4.0 * h) / dz) + 1, dtype=torch.float64, device=dev) * dz
        d2 = ((rn[:, 0] - p[0]) ** 2 + (rn[:, 1] - p[1]) ** 2)[:, None] + (rn[:, 2:3] - zs[None, :]) ** 2
        q = d2.sqrt() / h
        w = torch.where(q < 2.0, (1.0 - 0.5 * q) ** 4 * (2.0 * q + 1.0), torch.zeros_like(q))
        s = m * 21.0 / (16.0 * math.pi * h**3) * w.sum(0)
        level = torch.nonzero(s >= 0.5 * RHO0)
        height.append(float(zs[level.max()]) if len(level) else 0.0)
    out = dict(pressure=np.array(pressure), height=np.array(height))
    if c.obstacle is not None:
        end = len(r) - int((kind == GATE).sum())
        ids = torch.arange(end - c.lattice_counts(LAYERS)[2], end, device=dev)
        lo, hi = r[ids].min(0).values - 2.0 * h, r[ids].max(0).values + 2.0 * h
        keep = ((r >= lo) & (r <= hi)).all(1)
        _, acc, _ = _derivatives(c, r[keep], u[keep], rho[keep], kind[keep], False) if bool((keep & fl).any()) else (
            0, torch.zeros((int(keep.sum()), 3), dtype=torch.float64, device=dev), 0)
        a = torch.zeros_like(r)
        a[keep] = acc
        out["force"] = (m * a[ids].sum(0)).cpu().numpy()
    return out


def exact(case, seed):
    if case["path"] == "mps":
        return _exact_mps(case, seed)
    parts = _wcsph_inputs(case, seed)
    passes = case["steps"] * (2 if case["integrator"] == "symplectic" else 1)
    if passes * sum(27.0 * (2.0 * p[0].h / p[0].dp) ** 3 * len(p[1]) for p in parts) > MAX_EXACT:
        return None
    pos, vel, prev, gauges = [], [], [], {}
    for c, r, u, rho, kind in parts:
        r, u, rho, up, rp = _advance(case, c, r, u, rho, kind)
        off = 0.0 if case["form"] == "fp64" else RHO0
        pos.append(torch.cat([r, torch.zeros_like(r[:, :1])], 1))
        vel.append(torch.cat([u, rho[:, None] - off], 1))
        prev.append(torch.cat([up, rp[:, None] - off], 1))
        if case["probes"]:
            gauges = _probe_values(c, r, u, rho, torch.from_numpy(kind).to(r.device))
    return dict(position=torch.cat(pos), velocity=torch.cat(vel), previous=torch.cat(prev), **gauges)
