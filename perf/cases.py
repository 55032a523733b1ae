"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes what a running program holds (a context
loaded with a state, its captured graph, its couplers), ``run`` is one pass through the public
entry points, and ``exact`` gives the same outputs from a plain 64-bit restatement of the method
(Eqs. 1-6, the axisymmetric walls, the gradients by complex-step differentiation).

The beds are body-centred lattices with vacancies, radii spread by +-0.2 % and positions jittered,
at the spacing where two neighbours touch with probability 1/2: about 7.4 list entries and 3.7
contacts per particle with overlaps of some micrometres, which is what a settled and sheared bed
holds, without the tens of thousands of steps that settling takes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1705_03850_gb300 import adjoint, dem, levels, workloads

GRID = workloads.GRID
OVERLAP_JITTER = 5e-4      # position jitter per axis, in radii
RADIUS_SPREAD = 2e-3       # relative
VACANCIES = 0.08


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # a small box stepped on its own: parameter studies, teaching, the smallest calls, where a
        # step is a chain of launches and waits (the fused steps, lanes by size)
        {"name": "box_1440", "kind": "bed", "n": 1440, "steps": 200, "graph": 100, "lanes": 0, "lmax": 32},
        # the coarse-grain silo in discharge: cone and cylinder walls, removal below the orifice
        {"name": "silo_23438", "kind": "silo", "n": 23438, "diameter": 5.6e-3, "steps": 200, "graph": 100, "lanes": 0},
        # the reference silo in discharge, stepped one launch per step
        {"name": "silo_187504", "kind": "silo", "n": 187504, "diameter": 2.8e-3, "steps": 100, "graph": 50, "lanes": 1},
        # the sheared bed, the headline workload
        {"name": "bed_1m", "kind": "bed", "n": 1_000_000, "steps": 100, "graph": 50, "lanes": 1, "lmax": 32},
        # a bed of an uneven size, four times as large, in short bursts between two outputs
        {"name": "bed_3999997", "kind": "bed", "n": 3_999_997, "steps": 50, "graph": 50, "lanes": 1, "lmax": 24},
        # a parameter study: independent boxes of mixed sizes and materials in one context
        {"name": "batch_48", "kind": "batch", "boxes": 48, "nmin": 2000, "nmax": 200_000, "steps": 50, "graph": 50,
         "lmax": 32},
        # calibration: gradients of energy and runout of 64 columns to E, e and mu
        {"name": "columns_64", "kind": "adjoint", "boxes": 64, "n": 10_000, "steps": 100, "checkpoint": 25},
        # a few small columns: the same path where the launches count
        {"name": "columns_4", "kind": "adjoint", "boxes": 4, "n": 1003, "steps": 50, "checkpoint": 10},
        # three nested levels of the chute, each at its own time step, coupled both ways
        {"name": "chute_3_levels", "kind": "chute", "length": 2.75, "width": 0.15, "bed": 0.15, "periods": 4},
        # the two-level silo: small levels, a coupling call every 15 steps
        {"name": "silo_2_levels", "kind": "silo2", "periods": 8},
        # forces of a given state, for a host program's own integrator or a restart: the state is
        # written, the lists are built, forces and torques read
        {"name": "forces_300007", "kind": "forces", "n": 300_007, "lmax": 32},
        # an output frame of a running bed: a few steps, positions and velocities to the host, fields on a grid
        {"name": "frame_500k", "kind": "frame", "n": 500_000, "steps": 10, "graph": 10, "cells": 40},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bed", "bed", "silo", "silo", "batch", "adjoint", "chute", "silo2", "forces", "frame"])
    if kind == "bed":
        n = _log(rng, 1000, 3_900_000)
        graph = rng.choice([10, 25, 50])
        return {"kind": kind, "n": n, "steps": graph * rng.randint(1, 4) if n < 900_000 else graph, "graph": graph,
                "lanes": 0 if n < 60_000 else 1, "lmax": rng.choice([20, 24, 32])}
    if kind == "silo":
        n = _log(rng, 5000, 300_000)
        return {"kind": kind, "n": n, "diameter": round(2.8e-3 * (187504 / n) ** (1 / 3) * rng.uniform(0.9, 1.1), 5),
                "steps": 50 * rng.randint(1, 3), "graph": 50, "lanes": rng.choice([0, 0, 1])}
    if kind == "batch":
        return {"kind": kind, "boxes": rng.randint(3, 60), "nmin": _log(rng, 600, 5000),
                "nmax": _log(rng, 20_000, 150_000), "steps": 25 * rng.randint(1, 2), "graph": 25, "lmax": rng.choice([24, 32])}
    if kind == "adjoint":
        k = rng.choice([5, 10, 20])
        return {"kind": kind, "boxes": _log(rng, 1, 48), "n": _log(rng, 500, 9000), "steps": k * rng.randint(2, 4),
                "checkpoint": k}
    if kind == "chute":
        return {"kind": kind, "length": round(rng.uniform(1.5, 2.7), 2), "width": round(rng.uniform(0.1, 0.15), 3),
                "bed": round(rng.uniform(0.1, 0.15), 3), "periods": rng.randint(1, 4)}
    if kind == "silo2":
        return {"kind": kind, "periods": rng.randint(2, 8)}
    if kind == "forces":
        return {"kind": kind, "n": _log(rng, 3000, 900_000), "lmax": rng.choice([20, 24, 32])}
    return {"kind": kind, "n": _log(rng, 5000, 900_000), "steps": 10, "graph": 10, "cells": rng.randint(8, 60)}


def work(case):
    """Bytes and operations that a pass cannot do without.  Per particle and step: the state read and
    written (96 B), 4 B per list entry, the stored overlap of each contact read and written (24 B);
    about 190 operations per contact from each side and 120 for the rest.  What fits the 129 MB
    cache is read and written once a pass."""
    entries, contacts = 7.4, 3.7
    per_step, flops = 96 + 4 * entries + 24 * contacts, 190 * contacts + 120
    held = 96 + 4 * entries + 12 * contacts      # the state in two buffers

    def stepping(n, steps):
        return (n * per_step * steps if n * held > 129e6 else n * per_step), n * flops * steps
    kind = case["kind"]
    if kind in ("bed", "silo"):
        b, f = stepping(case["n"], case["steps"])
        return {"bytes": b + case["n"] * 72, "flops": f}
    if kind == "batch":
        n = int(np.sum(_sizes(case)))
        b, f = stepping(n, case["steps"])
        return {"bytes": b + n * 48, "flops": f}
    if kind == "adjoint":
        # forward, recomputation and reverse; the reverse pass also reads and writes the adjoint state
        # (96 B) and each contact's overlap adjoint, and every step's state comes back once from memory
        n, s = case["boxes"] * case["n"], case["steps"]
        return {"bytes": n * s * (held + 96 + 4 * entries + 24 * contacts), "flops": n * s * flops * 5}
    if kind == "chute":
        # FCC at contact: sqrt 2 / d^3 particles per volume; 6 of 12 neighbours touch
        b = f = 0
        for (L, _), d, s in zip(_chute_spans(case), (8e-3, 4e-3, 2e-3), (4, 8, 16)):
            n = math.sqrt(2) / d ** 3 * L * case["width"] * case["bed"]
            s *= case["periods"]
            b += n * (96 + 4 * 12 + 24 * 6) * (s if n * 168 > 129e6 else 1)
            f += n * (190 * 6 + 120) * s
        return {"bytes": b, "flops": f}
    if kind == "silo2":
        n, s = 23438 + 44000, 15 * case["periods"]
        return {"bytes": n * per_step, "flops": n * flops * s}
    n = case["n"]
    if kind == "forces":
        # the state in, forces and torques out, in double; 27 cells of about 2.2 particles searched
        return {"bytes": n * (11 * 8 + 6 * 8), "flops": n * (60 * 12 + 190 * contacts)}
    b, f = stepping(n, case["steps"])
    return {"bytes": b + n * 72 + 40 * case["cells"] ** 3, "flops": f + 20 * n}


# ------------------------------------------------------------------ inputs

def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _uniform(g, shape, a, b):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (b - a) + a


def _q(a):
    return torch.round(a / GRID) * GRID


def _f32(a):
    return a.to(torch.float32).to(torch.float64)


class System:
    """One system's inputs: float64 CUDA tensors x, v, w, r, m and its description."""

    def __init__(self, x, v, w, r, lo, hi, periodic, material, dt, floor=True, floor_v=(0.0, 0.0, 0.0), skin=2e-4,
                 walls=None, z_remove=-math.inf, axis=(0.0, 0.0)):
        self.lo, self.hi = tuple(float(a) for a in workloads.qgrid(lo)), tuple(float(a) for a in workloads.qgrid(hi))
        self.x, self.r = _q(x), _q(r)
        for a in range(3):
            if periodic[a]:
                L = self.hi[a] - self.lo[a]
                self.x[:, a] = self.lo[a] + torch.remainder(self.x[:, a] - self.lo[a], L)
        self.v, self.w = _f32(v), _f32(w)
        self.m = _f32(material.rho * (4.0 / 3.0) * math.pi * self.r ** 3)
        self.periodic, self.material, self.dt = periodic, material, float(np.float32(dt))
        self.g = (0.0, 0.0, float(np.float32(-9.81)))
        self.floor, self.floor_v, self.skin = floor, floor_v, float(workloads.qgrid(skin))
        self.walls, self.z_remove, self.axis = walls, z_remove, axis
        self.n = int(self.x.shape[0])

    def desc(self, capacity=None):
        m = self.material
        return dem.desc(n=self.n, lo=self.lo, hi=self.hi, periodic=self.periodic, dt=self.dt, skin=self.skin,
                        r_max=float(self.r.max()), E=m.E, nu=m.nu, e=m.e, mu=m.mu, mu_wall=m.mu_wall, rho=m.rho,
                        g=self.g, floor=self.floor, floor_v=self.floor_v, capacity=capacity)

    def state(self):
        return self.x, self.v, self.w, self.r, self.m


def _bcc(nx, ny, nz, a):
    """(2 nx ny nz, 3) sites of a body-centred lattice of constant a, lowest first."""
    ax = [torch.arange(k, device="cuda", dtype=torch.float64) for k in (nz, ny, nx)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    base = torch.stack([x, y, z], -1).reshape(nz, -1, 3) * a
    return torch.stack([base, base + 0.5 * a], 1).reshape(-1, 3)


def _thin(g, x, n, vacancies=VACANCIES):
    """n of the lowest sites x, with vacancies, in order."""
    x = x[: max(n, min(x.shape[0], int(math.ceil(n / (1 - vacancies)))))]
    return x[torch.sort(torch.randperm(x.shape[0], generator=g, device="cuda")[:n]).values]


def bed(n, seed, r=1e-3, material=None, dt=1e-6, shear=0.5, noise=0.02, spin=5.0, stream=0, open_sides=False):
    """n spheres on a dense lattice over a floor, periodic in x and y (or a free-standing column of
    square section), sheared by a floor that moves at `shear`."""
    g = _gen(seed, stream)
    a = 4.0 * r / math.sqrt(3.0)
    cells = n / (2 * (1 - VACANCIES))
    k = max(5, int(round((cells * (0.25 if open_sides else 1.0)) ** (1 / 3))))
    x = _thin(g, _bcc(k, k, int(math.ceil(cells / k ** 2)) + 1, a), n)
    top = float(x[:, 2].max())
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * noise
    v[:, 0] += shear * (1.0 - x[:, 2] / (top + r))
    w = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * spin
    x = x + _uniform(g, (n, 3), -OVERLAP_JITTER * r, OVERLAP_JITTER * r)
    rad = r * _uniform(g, (n,), 1 - RADIUS_SPREAD, 1 + RADIUS_SPREAD)
    x[:, 2] += r
    side = k * a
    if open_sides:
        margin = 10 * r
        x[:, :2] += margin + 0.25 * a
        box, per = side + 2 * margin, (False, False, False)
    else:
        x[:, :2] += 0.25 * a
        box, per = side, (True, True, False)
    return System(x, v, w, rad, (0, 0, 0), (box, box, top + 12 * r), per, material or workloads.Material(), dt,
                  floor_v=(float(np.float32(shear)), 0.0, 0.0), skin=0.2 * r, axis=(0.5 * box, 0.5 * box))


def silo(n, seed, d=2.8e-3, z_top=None, r_max=None, margin=None, height=0.5, stream=0):
    """Spheres packed in the cone and cylinder of the silo from the orifice up, the orifice open:
    n of them, or all below z_top within r_max of the axis."""
    g = _gen(seed, stream)
    z_o, r_o, R, h = 0.05, 0.02, 0.135, 0.2
    r, a = 0.5 * d, 2.0 * d / math.sqrt(3.0)
    m = int(math.ceil(R / a)) + 1
    x = _bcc(2 * m, 2 * m, int(math.ceil(((z_top or z_o + 2 * h) - z_o) / a)), a)
    x[:, :2] -= m * a
    x[:, 2] += z_o + r
    rho = torch.hypot(x[:, 0], x[:, 1])
    wall = torch.clamp(r_o + (R - r_o) * (x[:, 2] - z_o) / h, max=R)
    x = x[rho <= torch.clamp(wall, max=r_max or R) - r * math.hypot(1.0, (R - r_o) / h)]
    if z_top is not None:
        x = x[x[:, 2] <= z_top - d]
        n = int(x.shape[0] * (1 - VACANCIES))
    x = _thin(g, x, min(n, int(x.shape[0] * (1 - VACANCIES))))
    n = x.shape[0]
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64) * 0.02
    v[:, 2] -= 0.1
    x = x + _uniform(g, (n, 3), -OVERLAP_JITTER * r, OVERLAP_JITTER * r)
    rad = r * _uniform(g, (n,), 1 - RADIUS_SPREAD, 1 + RADIUS_SPREAD)
    box = margin or R + 2 * d
    return System(x, v, torch.zeros_like(v), rad, (-box, -box, 0.0), (box, box, height), (False, False, False),
                  workloads.SILO_MATERIAL, 1e-6, floor=False, skin=0.1 * d,
                  walls=workloads.silo_walls(z_o, closed=False), z_remove=z_o - 0.01)


def _sizes(case):
    u = (np.arange(case["boxes"]) + 0.5) / case["boxes"]
    return np.round(case["nmin"] * (case["nmax"] / case["nmin"]) ** u).astype(np.int64)


def _batch(case, seed):
    rng = np.random.default_rng(seed)
    sizes = rng.permutation(_sizes(case))
    return [bed(int(n), seed, material=workloads.Material(
        E=float(math.exp(rng.uniform(math.log(5e6), math.log(5e7)))), e=float(rng.uniform(0.5, 0.95)),
        mu=float(rng.uniform(0.2, 0.8))), stream=1 + k) for k, n in enumerate(sizes)]


def _columns(case, seed):
    mats = workloads.column_materials(case["boxes"], seed=seed)
    return [bed(case["n"], seed, material=mats[k], dt=5e-6, shear=0.0, noise=0.01, stream=1 + k, open_sides=True)
            for k in range(case["boxes"])]


def _chute_spans(case):
    L = case["length"]
    return (L, 0.0), (L * 0.128, L * 0.2), (L * 0.033, L * 0.25)


# ------------------------------------------------------------------ what a program has in hand

def _context(systems, lmax, capacity=None, stream=None):
    sim = dem.DEM([s.desc(capacity) for s in systems], max_neighbors=lmax, stream=stream)
    torch.cuda.synchronize()             # the inputs were made on the current stream
    sim.write_state(*(torch.cat(t) if len(systems) > 1 else t[0] for t in zip(*(s.state() for s in systems))))
    for k, s in enumerate(systems):
        if s.walls is not None:
            sim.set_walls(k, s.axis, s.walls, s.z_remove)
    torch.cuda.synchronize()             # ... and are let go here
    return sim


def _systems(case, seed):
    kind = case["kind"]
    if kind in ("bed", "forces", "frame"):
        return [bed(case["n"], seed)]
    if kind == "silo":
        return [silo(case["n"], seed, d=case["diameter"])]
    if kind == "batch":
        return _batch(case, seed)
    return _columns(case, seed)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("bed", "silo", "batch", "frame"):
        st["sim"] = sim = _context(_systems(case, seed), case.get("lmax", 24))
        if case.get("lanes", 1) != 1:
            sim.set_step_lanes(case["lanes"])
        sim.set_graph(case["graph"])
        if kind == "frame":
            st["edge"] = sim.info()["hi"][0] / case["cells"]
    elif kind == "adjoint":
        systems = _systems(case, seed)
        st["sim"] = _context(systems, 16)
        st["state"] = [torch.cat(t) for t in zip(*(s.state() for s in systems))]
        st["params"] = torch.tensor([[s.material.E, s.material.e, s.material.mu] for s in systems], dtype=torch.float64)
        st["axis"] = np.array([s.axis for s in systems])
        st["weights"] = torch.ones((case["boxes"], 2), dtype=torch.float64)
    elif kind == "forces":
        s = bed(case["n"], seed)
        st["sim"], st["state"] = _context([s], case["lmax"]), s.state()
    elif kind == "chute":
        (L0, _), (L1, x1), (L2, x2) = _chute_spans(case)
        lv, specs = workloads.chute(length=L0, width=case["width"], height=case["bed"] + 0.06, bed=case["bed"],
                                    regions=((x1, L1), (x2, L2)), seed=seed, interval=16, multirate=True, gap=0.0)
        ctx = []
        for k, wl in enumerate(lv):
            d = dem.DEM([dem.desc_from_workload(wl, capacity=None if k == 0 else wl.n + 60_000)], max_neighbors=24,
                        stream=torch.cuda.Stream())
            v = wl.v.copy()
            v[:, 0] += wl.meta["u0"]
            d.write_state(wl.x, v, wl.w, wl.r, wl.m)
            ctx.append(d)
        st["levels"], st["hierarchy"] = ctx, levels.Hierarchy(ctx, specs)
    else:
        _, _, spec = workloads.silo_two_level(seed=seed)
        coarse = silo(23438, seed, d=5.6e-3)
        fine = silo(0, seed, z_top=0.15, r_max=0.08, margin=0.09, height=0.18, stream=1)
        ctx = [_context([coarse], 24, stream=torch.cuda.Stream()),
               _context([fine], 24, capacity=fine.n + 100_000, stream=torch.cuda.Stream())]
        st["levels"], st["hierarchy"] = ctx, levels.Hierarchy(ctx, [spec])
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("bed", "silo", "batch"):
        sim = st["sim"]
        sim.step(case["steps"])
        out = {"x": sim.read(dem.POS, host=False), "v": sim.read(dem.VEL, host=False)}
        if kind != "batch":
            out["w"] = sim.read(dem.OMEGA, host=False)
        return out
    if kind == "frame":
        sim, k = st["sim"], case["cells"]
        sim.step(case["steps"])
        return {"x": sim.read(dem.POS), "v": sim.read(dem.VEL), "fields": sim.grid_fields((0.0, 0.0, 0.0), st["edge"], (k, k, k))}
    if kind == "forces":
        sim = st["sim"]
        sim.write_state(*st["state"])
        return {"force": sim.read(dem.FORCE, host=False), "torque": sim.read(dem.TORQUE, host=False)}
    if kind == "adjoint":
        p = st["params"].clone().requires_grad_()
        obs = adjoint.rollout(p, st["sim"], st["state"], case["steps"], case["checkpoint"], st["axis"])
        (grad,) = torch.autograd.grad(obs, p, st["weights"])
        return {"observables": obs.detach(), "dE": grad[:, 0], "de": grad[:, 1], "dmu": grad[:, 2]}
    st["hierarchy"].advance(case["periods"])
    here = torch.cuda.current_stream()
    out = {}
    for k, lv in enumerate(st["levels"]):       # each level's outputs come from its own stream
        lv.stream.wait_stream(here)
        out[k] = {"x": lv.read(dem.POS, host=False), "v": lv.read(dem.VEL, host=False)}
        here.wait_stream(lv.stream)
    if kind == "silo2":
        out["removed"] = [lv.wall_removed()[1] for lv in st["levels"]]
    return out


# ------------------------------------------------------------------ the same in 64 bits

def _pairs(s, margin):
    """Index pairs i, j closer than the sum of the largest radii plus the margin (cell lists)."""
    x, n = s.x, s.n
    cut = 2 * float(s.r.max()) + margin
    lo, hi = torch.tensor(s.lo, device="cuda", dtype=torch.float64), torch.tensor(s.hi, device="cuda", dtype=torch.float64)
    nc = [max(1, int((s.hi[a] - s.lo[a]) / cut)) for a in range(3)]
    size = torch.tensor(nc, device="cuda")
    c = torch.minimum(((x - lo) / (hi - lo) * size).floor().long().clamp(min=0), size - 1)
    order = torch.argsort((c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0], stable=True)
    c = c[order]
    code = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    count = torch.bincount(code, minlength=nc[0] * nc[1] * nc[2])
    start = torch.cumsum(count, 0) - count
    most, me = int(count.max()), torch.arange(n, device="cuda")
    I, J = [], []
    for k in range(13, 27):                      # the cell itself and half of its neighbours
        off = [k % 3 - 1, (k // 3) % 3 - 1, k // 9 - 1]
        ok, cc = torch.ones(n, dtype=torch.bool, device="cuda"), []
        for a in range(3):
            t = c[:, a] + off[a]
            if s.periodic[a]:
                t = torch.remainder(t, nc[a])
            else:
                ok &= (t >= 0) & (t < nc[a])
                t = t.clamp(0, nc[a] - 1)
            cc.append(t)
        o = (cc[2] * nc[1] + cc[1]) * nc[0] + cc[0]
        for t in range(most):
            sel = ok & (t < count[o]) & ((start[o] + t > me) if k == 13 else ok)
            i, j = order[me[sel]], order[(start[o] + t)[sel]]
            dx = x[i] - x[j]
            for a in range(3):
                if s.periodic[a]:
                    L = s.hi[a] - s.lo[a]
                    dx[:, a] -= L * torch.round(dx[:, a] / L)
            near = (dx * dx).sum(1) < cut * cut
            I.append(i[near])
            J.append(j[near])
    return torch.cat(I), torch.cat(J)


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _law(p, mu, delta, n, R, meff, vr, rw, xi, dt):
    """Force and tangential force of Eqs. 3-6 on the first body of each contact, and its new overlap."""
    root = torch.sqrt(R * delta)
    kn, kt = p["kn"] * root, p["kt"] * root
    gn, gt = p["nbeta"] * torch.sqrt(5 * meff * kn), p["nbeta"] * torch.sqrt(10 / 3 * meff * kt)
    vc = vr - torch.linalg.cross(rw, n)
    vt = vc - _dot(vc, n) * n
    fn = kn * delta - gn * _dot(vr, n)
    xr = xi - _dot(xi, n) * n
    l0, l1 = _dot(xi, xi), _dot(xr, xr)
    some = l1.real > 0
    xi = torch.where(some, torch.sqrt(l0 / torch.where(some, l1, torch.ones_like(l1))) * xr, torch.zeros_like(xr))
    xi = xi + dt * vt
    ft = -kt * xi - gt * vt
    ft2, lim = _dot(ft, ft), mu * torch.where(fn.real < 0, -fn, fn)
    slip = ft2.real > (lim * lim).real
    cut = lim / torch.sqrt(torch.where(slip, ft2, torch.ones_like(ft2))) * ft
    xi = torch.where(slip, -(cut + gt * vt) / kt, xi)
    ft = torch.where(slip, cut, ft)
    return fn * n + ft, ft, xi


class Exact:
    """The method in 64 bits for one system; `kind` complex with a step in one parameter gives derivatives."""

    def __init__(self, s, kind=torch.float64, step=None, margin=None):
        self.s, self.kind = s, kind
        m = s.material
        par = {"E": m.E, "e": m.e, "mu": m.mu}
        if step:
            par[step] = par[step] + 1e-30j
        par = {k: torch.tensor(v, dtype=kind, device="cuda") for k, v in par.items()}
        le = torch.log(par["e"])
        self.p = {"kn": 4 / 3 * par["E"] / (2 * (1 - m.nu ** 2)), "kt": 8 * par["E"] / (4 * (2 - m.nu) * (1 + m.nu)),
                  "nbeta": -le / torch.sqrt(le * le + math.pi ** 2)}
        self.mu = par["mu"]
        self.mu_w = par["mu"] if m.mu_wall is None else m.mu_wall
        self.x, self.v, self.w = (t.to(kind) for t in (s.x, s.v, s.w))
        self.r, self.m = s.r[:, None], s.m[:, None]
        self.i, self.j = _pairs(s, margin if margin is not None else s.skin)
        self.xi = torch.zeros((self.i.shape[0], 3), dtype=kind, device="cuda")
        self.nw = (1 if s.floor else 0) + (len(s.walls) - 1 if s.walls is not None else 0)
        self.wxi = torch.zeros((self.nw, s.n, 3), dtype=kind, device="cuda")

    def _walls(self):
        """Overlap, normal and wall velocity of every particle with every wall."""
        s, x = self.s, self.x
        zero = torch.zeros_like(x[:, :1])
        if s.floor:
            up = torch.zeros_like(x)
            up[:, 2] = 1
            yield self.r - (x[:, 2:] - s.lo[2]), up, torch.tensor(s.floor_v, dtype=self.kind, device="cuda")
        if s.walls is not None:
            ex = torch.stack([x[:, 0] - s.axis[0], x[:, 1] - s.axis[1]], 1)
            rho = torch.sqrt(_dot(ex, ex))
            er = ex / torch.where(rho.real > 0, rho, torch.ones_like(rho))
            for (r0, z0), (r1, z1) in zip(s.walls[:-1], s.walls[1:]):
                dr, dz = float(r1 - r0), float(z1 - z0)
                t = (((rho - r0) * dr + (x[:, 2:] - z0) * dz) / (dr * dr + dz * dz)).clamp(0, 1)
                a, b = rho - (r0 + t * dr), x[:, 2:] - (z0 + t * dz)
                dist = torch.sqrt(a * a + b * b)
                yield self.r - dist, torch.cat([a / dist * er, b / dist], 1), zero

    def forces(self, dt):
        """F and T at the current state, and the overlaps advanced by dt."""
        s, i, j = self.s, self.i, self.j
        F = self.m * torch.tensor(s.g, dtype=self.kind, device="cuda")
        T = torch.zeros_like(F)
        dx = self.x[i] - self.x[j]
        for a in range(3):
            if s.periodic[a]:
                L = s.hi[a] - s.lo[a]
                dx[:, a] -= L * torch.round(dx[:, a].real / L)
        d2 = _dot(dx, dx)
        k = (d2.real < (self.r[i] + self.r[j]) ** 2)[:, 0].nonzero()[:, 0]
        i, j, dx, d2 = i[k], j[k], dx[k], d2[k]
        dist = torch.sqrt(d2)
        n = dx / dist
        ri, rj, mi, mj = self.r[i], self.r[j], self.m[i], self.m[j]
        f, ft, x1 = _law(self.p, self.mu, ri + rj - dist, n, ri * rj / (ri + rj), mi * mj / (mi + mj),
                         self.v[i] - self.v[j], ri * self.w[i] + rj * self.w[j], self.xi[k], dt)
        t = torch.linalg.cross(n, ft)
        F.index_add_(0, i, f).index_add_(0, j, -f)
        T.index_add_(0, i, -ri * t).index_add_(0, j, -rj * t)
        xi = torch.zeros_like(self.xi)
        xi[k] = x1
        wxi = torch.zeros_like(self.wxi)
        for q, (delta, n, vw) in enumerate(self._walls()):
            k = (delta.real > 0)[:, 0].nonzero()[:, 0]
            n, r = n[k], self.r[k]
            f, ft, x1 = _law(self.p, self.mu_w, delta[k], n, r, self.m[k], self.v[k] - (vw if vw.dim() == 1 else 0),
                             r * self.w[k], self.wxi[q][k], dt)
            F.index_add_(0, k, f)
            T.index_add_(0, k, -r * torch.linalg.cross(n, ft))
            wxi[q][k] = x1
        return F, T, xi, wxi

    def run(self, steps):
        """Steps of velocity Verlet; then x, v, w at the last step (the half kick completed)."""
        s, dt, inertia = self.s, self.s.dt, 0.4 * self.m * self.r ** 2
        for n in range(steps + 1):
            F, T, xi, wxi = self.forces(dt if n else 0.0)
            kick = 0.5 * dt if n in (0, steps) else dt
            if n == 0 and steps == 0:
                kick = 0.0
            self.v = self.v + kick * F / self.m
            self.w = self.w + kick * T / inertia
            if n < steps:
                self.xi, self.wxi = xi, wxi
                self.x = self.x + dt * self.v
        self.F, self.T = F, T
        return self

    def wrapped(self):
        x = self.x.clone()
        for a in range(3):
            if self.s.periodic[a]:
                x[:, a] = self.s.lo[a] + torch.remainder(x[:, a] - self.s.lo[a], self.s.hi[a] - self.s.lo[a])
        return x

    def observables(self):
        s = self.s
        ke = (0.5 * self.m * _dot(self.v, self.v) + 0.2 * self.m * self.r ** 2 * _dot(self.w, self.w)).sum()
        e = self.x[:, :2] - torch.tensor(s.axis, dtype=torch.float64, device="cuda")
        k = int(torch.argmax((e.real ** 2).sum(1)))
        return ke, torch.sqrt((e[k] * e[k]).sum())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("chute", "silo2"):
        # a plain restatement of the insertion and its random draws, the stress controllers and the
        # removal, call by call, takes minutes
        return None
    if kind == "adjoint":
        # three complex rollouts of every column: about 20 s for some 30,000 particle-steps a column
        if case["boxes"] * case["steps"] > 2000:
            return None
        obs, grad = [], []
        for s in _columns(case, seed):
            d = []
            for name in ("E", "e", "mu"):
                o = Exact(s, torch.complex128, name).run(case["steps"]).observables()
                d.append(float((o[0] + o[1]).imag) / 1e-30)
            obs.append([float(t.real) for t in o])
            grad.append(d)
        g = torch.tensor(grad, dtype=torch.float64)
        return {"observables": torch.tensor(obs, dtype=torch.float64), "dE": g[:, 0], "de": g[:, 1], "dmu": g[:, 2]}
    done = [Exact(s).run(case.get("steps", 0)) for s in _systems(case, seed)]
    if kind == "forces":
        return {"force": done[0].F, "torque": done[0].T}
    out = {"x": torch.cat([e.wrapped() for e in done]), "v": torch.cat([e.v for e in done])}
    if kind == "frame":
        s, k = done[0].s, case["cells"]
        h = s.hi[0] / k
        c = torch.floor(out["x"] / h).long()
        ok = ((c >= 0) & (c < k)).all(1)
        c = c[ok]
        cell = (c[:, 2] * k + c[:, 1]) * k + c[:, 0]
        val = torch.cat([4 / 3 * math.pi * s.r[ok, None] ** 3 / h ** 3, s.m[ok, None], s.m[ok, None] * out["v"][ok]], 1)
        f = torch.zeros((k ** 3, 5), dtype=torch.float64, device="cuda").index_add_(0, cell, val)
        f[:, 2:] = torch.where(f[:, 1:2] > 0, f[:, 2:] / f[:, 1:2].clamp(min=1e-300), torch.zeros_like(f[:, 2:]))
        out["fields"] = f.reshape(k, k, k, 5)
        return out
    if kind != "batch":
        out["w"] = torch.cat([e.w for e in done])
    return out
