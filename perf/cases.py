"""Timed workloads of the Bloch-Torrey lattice solver, through its public calls.

Each case is one simulation job as a user's program runs it: a geometry and
its membranes are set once (``prepare``), and a pass (``run``) is the whole
call -- set-up of the run, every time step, the signal and what else the call
returns.  The kinds and what they stand for:

``free``      verification against exp(-bD): small uniform periodic grids, the
              schedule repeated for several b-values with a plain run each
``plain``     one gradient direction on a permeable cylinder or sphere pack,
              signal and magnetisation field
``specimen``  a specimen in a box with mirroring walls, edges of any length
``tissue``    the large tissue model: Voronoi cells, extracellular band and
              vessels, mirroring walls, three orthogonal directions in a batch
``batch``     many directions and b-values on one shared geometry plus sphere
              packs of uneven size (with their fields), one batched run
``protocol``  a protocol that mixes diffusion times: batched members with their
              own waveforms, echoes and field outputs on packs of any edge
``gradient``  batched adjoint: signal and its derivatives for many directions
``fit``       one objective evaluation of a microstructure fit through autograd
``ogse``      an oscillating gradient (waveform values other than 0 and +-1)
              with the signal recorded after every step and the final field
``links``     membranes at their exact positions on the links, 3-D
``slice``     the 2-D lattice on a large slice (the paper's 1000 x 1000 grids)
``study2d``   the paper's 2-D membrane-placement study: small grid, many steps

The geometries are seeded jittered lattices of bodies built with torch on the
device, so inputs are quick to make.  ``exact`` is the same scheme written
plainly in complex128 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1907_00908_gb300 import lbmbt
from paper_1907_00908_gb300.autograd import signal

INF = math.inf
E = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1))


def _case(kind, name=None, **kw):
    c = {"kind": kind, **kw}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest: 32^3 free diffusion, the full schedule, five b-values
        _case("free", "free32", nx=32, ny=32, nz=32, steps=2000, runs=5, series=False),
        # two-phase permeable cylinders, one direction, 128^3
        _case("plain", "cylinders128", body="cylinders", nx=128, ny=128, nz=128, steps=1280),
        # odd edges, mirroring walls on two axes
        _case("specimen", "specimen_odd", nx=117, ny=90, nz=75, steps=480),
        # the large tissue model: 512^3, three directions (a slice of its schedule)
        _case("tissue", "tissue512", nx=512, ny=512, nz=512, steps=48),
        # many directions on one 128^3 geometry plus uneven packs
        _case("batch", "batch128", n=128, members=40, packs=4, pack_min=48, pack_max=160, steps=48),
        # mixed diffusion times on packs with odd edges
        _case("protocol", "protocol_uneven", geometries=4, edge_min=57, edge_max=110, per=4, steps=160),
        # the gradient workload: 96^3 sphere pack, checkpoint every 64 steps
        _case("gradient", "gradient96", n=96, members=10, steps=128, every=64),
        # a fit's objective and gradient on a small voxel
        _case("fit", "fit48", n=48, steps=400, every=64),
        # oscillating gradient, every step's signal
        _case("ogse", "ogse160", nx=160, ny=144, nz=120, steps=128, periods=4),
        # exact membrane positions on the links
        _case("links", "links192", n=192, steps=64),
        # 2-D lattice, the paper's grid size
        _case("slice", "slice1000", nx=1000, ny=1000, steps=800),
        # 2-D membrane placement study, 200 x 200
        _case("study2d", "study200", n=200, steps=4000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["free", "plain", "specimen", "tissue", "batch", "protocol", "gradient", "fit", "ogse",
                       "links", "slice", "study2d"])
    if kind == "free":
        return _case(kind, nx=rng.randint(16, 48), ny=rng.randint(16, 48), nz=rng.randint(16, 48),
                     steps=rng.randint(500, 2000), runs=rng.randint(1, 5), series=rng.random() < 0.3)
    if kind == "plain":
        return _case(kind, body=rng.choice(["cylinders", "spheres"]), nx=rng.choice([rng.randint(40, 176), 16 * rng.randint(3, 11)]),
                     ny=rng.randint(40, 160), nz=rng.randint(24, 160), steps=_log(rng, 64, 1024))
    if kind == "specimen":
        return _case(kind, nx=rng.randint(33, 200), ny=rng.randint(33, 160), nz=rng.randint(20, 130),
                     steps=_log(rng, 64, 600))
    if kind == "tissue":
        return _case(kind, nx=16 * rng.randint(10, 28), ny=rng.randint(140, 400), nz=rng.randint(96, 320),
                     steps=rng.randint(12, 40))
    if kind == "batch":
        return _case(kind, n=16 * rng.randint(4, 9), members=_log(rng, 6, 40),
                     packs=rng.randint(1, 4), pack_min=rng.randint(40, 100), pack_max=rng.randint(100, 160),
                     steps=rng.randint(16, 48))
    if kind == "protocol":
        return _case(kind, geometries=rng.randint(1, 4), edge_min=rng.randint(40, 80), edge_max=rng.randint(80, 120),
                     per=rng.randint(1, 5), steps=rng.randint(48, 200))
    if kind == "gradient":
        return _case(kind, n=rng.choice([rng.randint(48, 112), 16 * rng.randint(3, 7)]), members=rng.randint(1, 8),
                     steps=rng.randint(40, 128), every=rng.choice([8, 16, 32, 64]))
    if kind == "fit":
        return _case(kind, n=rng.choice([rng.randint(24, 72), 16 * rng.randint(2, 4)]), steps=rng.randint(64, 400),
                     every=rng.choice([16, 64]))
    if kind == "ogse":
        return _case(kind, nx=rng.randint(60, 176), ny=rng.randint(60, 160), nz=rng.randint(40, 140),
                     steps=rng.randint(32, 160), periods=rng.randint(1, 6))
    if kind == "links":
        return _case(kind, n=rng.randint(64, 200), steps=rng.randint(16, 80))
    if kind == "slice":
        return _case(kind, nx=rng.randint(300, 1500), ny=rng.randint(300, 1200), steps=_log(rng, 64, 800))
    return _case("study2d", n=rng.randint(60, 260), steps=_log(rng, 500, 4000))


# ------------------------------------------------------------------ geometry

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lattice(shape, dx, pitch, gen, ndim):
    """Jittered lattice of body centres in a periodic box: cells per axis
    (x, y, z), pitches (um), centres [cz, cy, cx, 3]."""
    nz, ny, nx = shape
    L = [nx * dx, ny * dx, nz * dx]
    c = [max(3, int(round(v / pitch))) for v in L]
    if ndim == 2:
        c[2] = 1
    p = [L[a] / c[a] for a in range(3)]
    j = torch.rand((c[2], c[1], c[0], 3), generator=gen, dtype=torch.float64) - 0.5
    idx = torch.stack(torch.meshgrid(*[torch.arange(n, dtype=torch.float64) for n in (c[2], c[1], c[0])],
                                     indexing="ij"), -1).flip(-1)
    cen = (idx + 0.5 + 0.1 * j) * torch.tensor(p, dtype=torch.float64)
    return c, p, L, cen


def _candidates(shape, dx, c, p, cen, z0, z1, ndim):
    """For the planes z0..z1: the nearby cells' flat index and the vectors from
    the node to their centres (periodic images), one candidate at a time."""
    nz, ny, nx = shape
    dev = cen.device
    pos = [torch.arange(nx, device=dev, dtype=torch.float32) * dx, torch.arange(ny, device=dev, dtype=torch.float32) * dx,
           torch.arange(z0, z1, device=dev, dtype=torch.float32) * dx]
    cell = [torch.floor(pos[a] / p[a]).long() for a in range(3)]
    cf = cen.reshape(-1, 3).float()
    dz_range = (0,) if ndim == 2 else (-1, 0, 1)
    for oz in dz_range:
        for oy in (-1, 0, 1):
            for ox in (-1, 0, 1):
                off = (ox, oy, oz)
                w = [cell[a] + off[a] for a in range(3)]
                sh = [torch.div(w[a], c[a], rounding_mode="floor").float() * (c[a] * p[a]) for a in range(3)]
                k = [torch.remainder(w[a], c[a]) for a in range(3)]
                flat = (k[2][:, None, None] * c[1] + k[1][None, :, None]) * c[0] + k[0][None, None, :]
                v = cf[flat]
                dxv = v[..., 0] + sh[0][None, None, :] - pos[0][None, None, :]
                dyv = v[..., 1] + sh[1][None, :, None] - pos[1][None, :, None]
                dzv = v[..., 2] + sh[2][:, None, None] - pos[2][:, None, None] if ndim == 3 else torch.zeros_like(dxv)
                yield flat, dxv, dyv, dzv


def _bodies(shape, dx, seed, kind):
    """Pack of spheres or z-aligned cylinders: labels (0 outside, cell + 1
    inside), phase per label, centres and radii."""
    gen = torch.Generator().manual_seed(seed)
    ndim = 2 if kind == "cylinders" else 3
    c, p, L, cen = _lattice(shape, dx, 6.0, gen, ndim)
    n = cen[..., 0].numel()
    half = 0.5 * min(p[:ndim])
    rad = half * (0.72 + 0.17 * torch.rand(n, generator=gen, dtype=torch.float64))   # neighbours are >= 1.8 half apart
    dev = _dev()
    cen, rad = cen.to(dev), rad.to(dev)
    lab = torch.zeros(shape, dtype=torch.int32, device=dev)
    rf = rad.float()
    for z0 in range(0, shape[0], 64):
        z1 = min(shape[0], z0 + 64)
        for flat, dxv, dyv, dzv in _candidates(shape, dx, c, p, cen, z0, z1, ndim):
            d2 = dxv * dxv + dyv * dyv + dzv * dzv
            lab[z0:z1] = torch.where(d2 < rf[flat] ** 2, flat.int() + 1, lab[z0:z1])
    pol = np.ones(n + 1, np.uint8)
    pol[0] = 0
    return lab, pol, cen.reshape(-1, 3), rad, L


def _tissue(shape, dx, seed):
    """Voronoi cells (phase 0), the band between them (phase 1) and four
    vessel tubes along z (phase 2)."""
    gen = torch.Generator().manual_seed(seed)
    c, p, L, cen = _lattice(shape, dx, 8.0, gen, 3)
    n = cen[..., 0].numel()
    dev = _dev()
    cen = cen.to(dev)
    nz, ny, nx = shape
    lab = torch.empty(shape, dtype=torch.int32, device=dev)
    tubes = (torch.rand((4, 2), generator=gen) * torch.tensor([L[0], L[1]])).to(dev)
    xx = torch.arange(nx, device=dev) * dx
    yy = torch.arange(ny, device=dev) * dx
    vessel = torch.zeros((ny, nx), dtype=torch.int32, device=dev)
    for t in range(4):
        vessel[((xx[None, :] - tubes[t, 0]) ** 2 + (yy[:, None] - tubes[t, 1]) ** 2) < 9.0] = n + 2 + t
    for z0 in range(0, nz, 32):
        z1 = min(nz, z0 + 32)
        d1 = torch.full((z1 - z0, ny, nx), INF, device=dev)
        d2 = d1.clone()
        own = torch.zeros(d1.shape, dtype=torch.int32, device=dev)
        for flat, dxv, dyv, dzv in _candidates(shape, dx, c, p, cen, z0, z1, 3):
            d = dxv * dxv + dyv * dyv + dzv * dzv
            near = d < d1
            d2 = torch.where(near, d1, torch.minimum(d2, d))
            own = torch.where(near, flat.int(), own)
            d1 = torch.where(near, d, d1)
        l = torch.where(torch.sqrt(d2) - torch.sqrt(d1) < 0.55, torch.full_like(own, n), own)
        lab[z0:z1] = torch.where(vessel[None] > 0, vessel[None] - 1, l)
    pol = np.zeros(n + 5, np.uint8)
    pol[n] = 1
    pol[n + 1:] = 2
    return lab, pol


def _positions(lab, cen, rad, L, dx, ndim):
    """Where each membrane cuts its link, float32 [6, nz, ny, nx] in dx, 0.5
    off the membranes (the body one end lies in; between two bodies the
    lower-labelled one)."""
    nz, ny, nx = lab.shape
    out = torch.full((6, nz, ny, nx), 0.5, dtype=torch.float32, device=lab.device)
    box = torch.tensor(L, dtype=torch.float64, device=lab.device)
    for j in range(6):
        e = E[j + 1]
        a = j // 2
        if a == 2 and (nz == 1 or ndim == 2):
            continue
        nb = torch.roll(lab, -e[a], dims=2 - a)
        zi, yi, xi = torch.nonzero(nb != lab, as_tuple=True)
        la, lb = lab[zi, yi, xi].long(), nb[zi, yi, xi].long()
        k = torch.where((la > 0) & (lb > 0), torch.minimum(la, lb), torch.maximum(la, lb)) - 1
        v = torch.stack([xi, yi, zi], 1).double() * dx - cen[k]
        v -= box * torch.round(v / box)
        ev = torch.tensor(e, dtype=torch.float64, device=lab.device)
        if ndim == 2:
            v[:, 2] = 0.0
        b = v @ ev
        disc = torch.sqrt(torch.clamp(b * b - (v * v).sum(1) + rad[k] ** 2, min=0.0))
        t1, t2 = -b - disc, -b + disc
        t = torch.where((t1 > 0) & (t1 < dx), t1, t2) / dx
        out[j][zi, yi, xi] = torch.clamp(t, 1e-3, 1 - 1e-3).float()
    return out


def _directions(n, seed):
    v = np.random.default_rng(seed).normal(size=(n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _pgse(steps):
    """Waveform of a pulse pair filling the schedule: a quarter on, half off
    (with the ends of the pulses inside), a quarter reversed."""
    n = max(1, steps // 4)
    f = np.zeros(steps)
    f[:n] = 1.0
    f[steps - n:] = -1.0
    return f


# ------------------------------------------------- the physics of every kind

def _amplitude(s, r):
    """gamma G0 (rad/(um ms)) of a strong gradient system, less for long pulses
    so that signal is left at the echo."""
    on = float(np.sum(np.asarray(s["f"]) > 0)) * s["dt"]
    return min(0.4, 0.45 / on) * r.uniform(0.6, 1.0)


def _setting(case, seed):
    """Everything a kind fixes besides the grid: dx, dt, D, T2, kappa, faces,
    lattice, waveforms and the members (gradient vector, geometry, kappa)."""
    k = case["kind"]
    r = np.random.default_rng(1000 + seed)
    s = {"lattice": 0, "bc": (0, 0, 0), "wave": None}
    if k == "free":
        s.update(dx=1.0, dt=0.0125, D=[2.0], T2=[INF], kappa=INF)
        f = np.zeros(case["steps"])
        on = case["steps"] // 5
        f[:on] = 1.0
        f[case["steps"] - on:] = -1.0
        d, D = on * s["dt"], (case["steps"] - on) * s["dt"]
        b = np.linspace(0.0, 2.0, case["runs"] + 1)[1:] * r.uniform(0.8, 1.2)
        s["f"] = f
        s["members"] = [((math.sqrt(v / (d * d * (D - d / 3))), 0.0, 0.0), 0, INF) for v in b]
        return s
    if k in ("slice", "study2d"):
        s.update(lattice=1, dx=0.5, dt=0.0125 if k == "slice" else 0.02, D=[2.3, 1.0] if k == "slice" else [2.3, 1.5],
                 T2=[80.0, 50.0], kappa=0.05, f=_pgse(case["steps"]))
        if k == "slice":
            s["bc"] = (1, 1, 0)
            g = (_amplitude(s, r), 0.0, 0.0)
        else:
            d = _directions(1, seed)[0]
            a = _amplitude(s, r) / math.hypot(d[0], d[1])
            g = (a * d[0], a * d[1], 0.0)
        s["members"] = [(g, 0, s["kappa"])]
        return s
    if k == "tissue":
        s.update(dx=0.25, dt=0.0015625, D=[1.0, 2.5, 3.0], T2=[50.0, 80.0, 80.0], kappa=0.01, bc=(1, 1, 1),
                 f=_pgse(case["steps"]))
        a = _amplitude(s, r)
        s["members"] = [((a, 0.0, 0.0), 0, 0.01), ((0.0, a, 0.0), 0, 0.01), ((0.0, 0.0, a), 0, 0.01)]
        return s
    s.update(dx=0.5, dt=0.025 if k in ("fit", "gradient") else 0.00625, D=[2.0, 1.0], T2=[80.0, 50.0], kappa=0.02)
    f = _pgse(case["steps"])
    if k == "ogse":
        n = case["steps"]
        f = np.cos(2 * math.pi * case["periods"] * (np.arange(n) + 0.5) / n)
    s["f"] = f
    amp = _amplitude(s, r)
    if k == "specimen":
        s["bc"] = (1, 0, 1)
        s["members"] = [((amp, 0.0, 0.0), 0, 0.02)]
    elif k in ("plain", "ogse", "links", "fit"):
        d = _directions(1, seed)[0]
        s["members"] = [(tuple(amp * d), 0, 0.02)]
    elif k == "batch":
        m = [(tuple(amp * (0.2 + 0.8 * (i % 8) / 7) * v), 0, 0.02) for i, v in enumerate(_directions(case["members"], seed))]
        m += [(tuple(amp * v), 1 + i, float(r.uniform(0.0, 0.05)))
              for i, v in enumerate(_directions(case["packs"], seed + 1))]
        s["members"] = m
    elif k == "protocol":
        m, w = [], []
        dirs = _directions(case["geometries"] * case["per"], seed)
        for i, v in enumerate(dirs):
            m.append((tuple(amp * v), i // case["per"], 0.02))
            n = max(8, int(case["steps"] * (0.4 + 0.6 * ((i * 5) % 7) / 6)))
            w.append(_pgse(n) if n < case["steps"] else None)
        s["members"], s["wave"] = m, w
    elif k == "gradient":
        s["members"] = [(tuple(amp * v), 0, 0.02) for v in _directions(case["members"], seed)]
    return s


def _edges(n, lo, hi):
    return [int(round(v)) for v in np.linspace(lo, hi, n)]


def _shapes(case):
    k = case["kind"]
    if k in ("free", "plain", "specimen", "tissue", "ogse"):
        return [(case["nz"], case["ny"], case["nx"])]
    if k == "slice":
        return [(1, case["ny"], case["nx"])]
    if k == "study2d":
        return [(1, case["n"], case["n"])]
    if k == "batch":
        return [(case["n"],) * 3] + [(e,) * 3 for e in _edges(case["packs"], case["pack_min"], case["pack_max"])]
    if k == "protocol":
        return [(e,) * 3 for e in _edges(case["geometries"], case["edge_min"], case["edge_max"])]
    return [(case["n"],) * 3]


def _geometries(case, seed, dx):
    """Per geometry: (labels on the device, phase per label, positions or None)."""
    k = case["kind"]
    out = []
    for i, sh in enumerate(_shapes(case)):
        if k == "free":
            out.append((torch.zeros(sh, dtype=torch.int32, device=_dev()), np.zeros(1, np.uint8), None))
        elif k == "tissue":
            out.append((*_tissue(sh, dx, seed), None))
        else:
            kind = case.get("body", "cylinders" if k in ("slice", "study2d", "links") or (k == "batch" and i == 0) else "spheres")
            lab, pol, cen, rad, L = _bodies(sh, dx, seed + 17 * i, kind)
            pos = _positions(lab, cen, rad, L, dx, 2 if kind == "cylinders" else 3) if k in ("links", "study2d") else None
            out.append((lab, pol, pos))
    return out


# ----------------------------------------------------------- prepare and run

def prepare(case, seed):
    s = _setting(case, seed)
    sol = lbmbt.Solver(0)
    if s["lattice"]:
        sol.set_option(lbmbt.OPT_LATTICE, 1)
    for i, (lab, pol, pos) in enumerate(_geometries(case, seed, s["dx"])):
        (sol.add_geometry if i else sol.set_geometry)(lab, pol, s["dx"], s["bc"])
        if pos is not None:
            sol.set_link_distances(pos, i)
    sol.set_phases(s["D"], s["T2"])
    sol.set_permeability(s["kappa"])
    sol.set_sequence(s["dt"], s["f"], s["members"][0][0])
    st = {"case": case, "sol": sol, "s": s}
    k = case["kind"]
    sizes = [int(np.prod(sh)) for sh in _shapes(case)]
    if k in ("free", "plain", "specimen", "ogse", "links", "slice", "study2d"):
        st["field"] = torch.zeros(sizes[0], dtype=torch.complex64, device="cuda")
    if k in ("tissue", "batch", "protocol", "gradient"):
        st["members"] = lbmbt.Solver.members([m[0] for m in s["members"]], [m[1] for m in s["members"]],
                                             [m[2] for m in s["members"]])
    if k in ("tissue", "batch", "protocol"):   # of the batch, the packs' fields
        st["fields"] = [torch.zeros(sizes[m[1]], dtype=torch.complex64, device="cuda") if k != "batch" or m[1] else None
                        for m in s["members"]]
    if k == "fit":
        st["params"] = [torch.tensor(s["D"], dtype=torch.float64, requires_grad=True),
                        torch.tensor(s["T2"], dtype=torch.float64, requires_grad=True),
                        torch.tensor(s["kappa"], dtype=torch.float64, requires_grad=True)]
    torch.cuda.synchronize()
    return st


def run(state):
    case, sol, s = state["case"], state["sol"], state["s"]
    k = case["kind"]
    if k == "free":
        out = {"Z": [], "series": []}
        for g, _, _ in s["members"]:
            sol.set_sequence(s["dt"], s["f"], g)
            r = sol.run(field=state["field"], series=case["series"])
            out["Z"].append(r["Z"])
            out["series"].append(r.get("series", np.zeros(0)))
        return {"Z": np.array(out["Z"]), "series": np.concatenate(out["series"]), "field": state["field"]}
    if k in ("plain", "specimen", "links", "slice", "study2d"):
        r = sol.run(field=state["field"])
        return {"Z": np.array([r["Z"]]), "field": state["field"]}
    if k == "ogse":
        r = sol.run(field=state["field"], series=True)
        return {"Z": np.array([r["Z"]]), "series": r["series"], "field": state["field"]}
    if k in ("tissue", "batch", "protocol"):
        r = sol.run_batch(state["members"], waveforms=s["wave"], fields=state["fields"])
        return {"Z": r["Z"], "S": r["S"], "fields": [f for f in state["fields"] if f is not None]}
    if k == "gradient":
        r = sol.grad_batch(state["members"], checkpoint_every=case["every"])
        return {"Z": r["Z"], "dD": r["dD"], "dT2": r["dT2"], "dkappa": r["dkappa"]}
    for p in state["params"]:
        p.grad = None
    S = signal(sol, *state["params"], checkpoint_every=case["every"])
    S.backward()
    return {"S": S.detach(), "dD": state["params"][0].grad, "dT2": state["params"][1].grad,
            "dkappa": state["params"][2].grad}


def _member_steps(case):
    """[(sites, steps)] of every run the pass makes."""
    sh = [int(np.prod(x)) for x in _shapes(case)]
    s = _setting(case, 0)
    out = []
    for i, (_, g, _) in enumerate(s["members"]):
        w = s["wave"][i] if s["wave"] else None
        out.append((sh[g], case["steps"] if w is None else len(w)))
    return out


def work(case):
    """The inputs of a pass are the geometry (a byte a site; four more bytes a
    cut link with positions, about 4 % of the links), its outputs the fields,
    signals and gradients; the populations between two steps are neither, so
    they are not counted.  Operations per site and step: reaction 8 a
    population, their sum 2, relaxation 6 (Q populations), and for the adjoint
    the step again, its transpose and the three sensitivities."""
    k = case["kind"]
    sizes = [int(np.prod(x)) for x in _shapes(case)]
    q = 5 if k in ("slice", "study2d") else 7
    ms = _member_steps(case)
    by = sum(sizes)
    if k in ("links", "study2d"):
        by += sum(sizes) * 6 * 0.04 * 4
    if k in ("free", "plain", "specimen", "ogse", "links", "slice", "study2d"):
        by += 8 * sizes[0]
    if k in ("tissue", "protocol"):
        by += sum(8 * n for n, _ in ms)
    if k == "batch":
        by += sum(8 * n for n in sizes[1:])
    if k == "ogse":
        by += 16 * case["steps"]
    ops = 16 * q * (3.5 if k in ("gradient", "fit") else 1.0)
    return {"bytes": int(by + 24 * len(ms)), "flops": int(ops * sum(n * t for n, t in ms))}


# ----------------------------------------------------- the scheme in 64 bits

def _cut(lab, bc):
    """memb[i]: the link from a node to node - e_i carries a membrane."""
    out = [None]
    for i in range(1, 7):
        a = (i - 1) // 2
        m = torch.roll(lab, E[i][a], dims=2 - a) != lab
        if bc[a]:
            m.select(2 - a, 0 if E[i][a] > 0 else -1).fill_(False)
        out.append(m)
    return out


def _pull(g, i, bc, gG, dx, F, dims):
    """Population i arriving at every node: streamed from node - e_i, with the
    phase of a periodic face or the image of a mirroring one."""
    a = (i - 1) // 2
    sgn = E[i][a]
    ib = i + 1 if i & 1 else i - 1
    dim = 2 - a
    v = torch.roll(g[i], sgn, dims=dim)
    if bc[a] == 0 and gG[a] == 0.0:
        return v
    v = v.clone()
    at = 0 if sgn > 0 else dims[a] - 1
    face = v.select(dim, at)
    if bc[a] == 0:
        ph = gG[a] * dims[a] * dx * F
        face.mul_(complex(math.cos(ph), math.sin(ph) * sgn))
    else:
        w = g[ib].select(dim, at)
        if gG[a] != 0.0:
            psi = gG[a] * dx * F * (-1.0 if sgn > 0 else 2 * dims[a] - 1.0)
            w = torch.conj(w) * complex(math.cos(psi), -math.sin(psi))
        face.copy_(w)
    return v


def _link_rule(g, i, dl, rho, bc, gG, dx, F, dims):
    """Membrane at dl (in dx) from the node on its link to node - e_i, normal
    to the link: the arriving population from the Dirichlet and Neumann
    relations of both sides joined by the flux rho (jump)."""
    ib = i + 1 if i & 1 else i - 1
    a = (i - 1) // 2
    e, dim = E[i][a], 2 - a

    def at(p, d):   # population p at node + d e_i, with the wrap phases
        v = torch.roll(g[p], -d * e, dims=dim)
        if gG[a] != 0.0:
            ph = gG[a] * dims[a] * dx * F
            c = torch.arange(dims[a], device=v.device) + d * e
            turn = torch.where(c < 0, 1.0, torch.where(c >= dims[a], -1.0, 0.0)).double() * ph
            sh = [1, 1, 1]
            sh[dim] = dims[a]
            v = v * torch.polar(torch.ones_like(turn), turn).reshape(sh)
        return v

    def coef(d):
        q, u = 1.0 / (2 * d + 1), 2 * d - 1
        return (1.0, -u * q, u * q, 2 * q), (2 * (d - 1), -u * u * q, 2 * u * q, (3 - 2 * d) * q)
    n, c = coef(dl)
    ns, cs = coef(1 - dl)
    den = c[3] * cs[3] + (c[3] * ns[3] + n[3] * cs[3]) * rho
    own, far = (g[ib], at(ib, 1), g[i]), (at(i, -1), at(i, -2), at(ib, -1))
    r = 0
    for j in range(3):
        r = r + own[j] * ((c[3] * cs[3] * n[j] + (cs[3] * n[3] * c[j] + ns[3] * c[3] * n[j]) * rho) / den)
        r = r + far[j] * (c[3] * n[3] * (ns[j] - cs[j]) * rho / den)
    return r


class _Exact:
    def __init__(self, lab, pol, pos, st):
        self.st, self.lab = st, lab
        nz, ny, nx = lab.shape
        self.dims = (nx, ny, nz)
        self.bc = st["bc"]
        self.phase = torch.as_tensor(pol.astype(np.int64), device=lab.device)[lab.long()]
        self.cut = _cut(lab, self.bc)
        self.pos = pos
        self.q = 5 if st["lattice"] else 7
        self.eps = 1.0 / 3 if st["lattice"] else 0.25
        self.w = [self.eps] + [self.eps / 2] * (self.q - 1)
        self.any = [None] + [bool(m.any()) for m in self.cut[1:]]
        dev = lab.device
        self.ax = [torch.arange(n, dtype=torch.float64, device=dev) for n in self.dims]

    def params(self, D, T2, kappa):
        dt, dx = self.st["dt"], self.st["dx"]
        om = 1.0 / (0.5 + dt * D / (self.eps * dx * dx))
        dec = torch.exp(-dt / T2)
        share = 1.0 if not torch.is_tensor(kappa) and math.isinf(kappa) else kappa / (kappa + self.eps * dx / (2 * dt))
        return om[self.phase], dec[self.phase], share, kappa

    def step(self, g, par, gG, f, F):
        om, dec, share, kappa = par
        st = self.st
        new = [g[0]]
        for i in range(1, self.q):
            ib = i + 1 if i & 1 else i - 1
            v = _pull(g, i, self.bc, gG, st["dx"], F, self.dims)
            if self.any[i] and not (not torch.is_tensor(kappa) and math.isinf(kappa)):
                h = g[ib] + share * (v - g[ib])
                if self.pos is not None:
                    a = (i - 1) // 2
                    e, dim = E[i][a], 2 - a
                    # half-link where node + e_i or node - 2 e_i lies in another compartment
                    use = self.cut[i] & ~self.cut[ib] & ~torch.roll(self.cut[i], e, dims=dim)
                    dl = self.pos[ib - 1].double()
                    rho = kappa * st["dt"] / (self.eps * st["dx"])
                    h = torch.where(use, _link_rule(g, i, dl, rho, self.bc, gG, st["dx"], F, self.dims), h)
                v = torch.where(self.cut[i], h, v)
            new.append(v)
        th = 0.0
        for a in range(3):
            if gG[a] != 0.0 and f != 0.0:
                sh = [1, 1, 1]
                sh[2 - a] = self.dims[a]
                th = th + (-gG[a] * st["dx"] * st["dt"] * f) * self.ax[a].reshape(sh)
        fac = dec * torch.polar(torch.ones_like(th), th) if torch.is_tensor(th) else dec
        new = [v * fac for v in new]
        M = sum(new[1:], new[0])
        return [v + om * (w * M - v) for v, w in zip(new, self.w)], M

    def run(self, D, T2, kappa, gG, f, series=False, grad=False):
        dev = self.lab.device
        par = self.params(D, T2, kappa)
        g = [torch.full(self.lab.shape, w, dtype=torch.complex128, device=dev) for w in self.w]
        F, ser, M = 0.0, [], None
        chunk = 8

        def advance(k0, k1, F, g, par):
            for k in range(k0, k1):
                g, M = self.step(g, par, gG, float(f[k]), F)
                F += float(f[k]) * self.st["dt"]
                if series:
                    ser.append(M.sum().item())
            return g, M, F
        for k0 in range(0, len(f), chunk):
            k1 = min(len(f), k0 + chunk)
            if grad:
                def fn(om, dec, share, *gg, k0=k0, k1=k1, F=F):
                    o, m, _ = advance(k0, k1, F, list(gg), (om, dec, share, par[3]))
                    return (*o, m)
                res = checkpoint(fn, *par[:3], *g, use_reentrant=False)
                g, M = list(res[:-1]), res[-1]
                F += float(np.sum(f[k0:k1])) * self.st["dt"]
            else:
                g, M, F = advance(k0, k1, F, g, par)
        return M, ser


def exact(case, seed):
    k = case["kind"]
    cost = sum(n * t for n, t in _member_steps(case)) * {"gradient": 5, "fit": 5, "links": 6, "study2d": 6}.get(k, 1)
    launches = case["steps"] * len(_member_steps(case))
    if cost > 6e9 or launches > 12000:
        return None
    st = _setting(case, seed)
    geo = _geometries(case, seed, st["dx"])
    dev = _dev()
    D = torch.tensor(st["D"], dtype=torch.float64, device=dev)
    T2 = torch.tensor(st["T2"], dtype=torch.float64, device=dev)
    solver, Z, series, fields = {}, [], [], []
    grads = {"dD": [], "dT2": [], "dkappa": []}
    S = []
    grad = k in ("gradient", "fit")
    for i, (gG, gi, kap) in enumerate(st["members"]):
        if gi not in solver:
            solver = {gi: _Exact(*geo[gi], st)}
        f = st["wave"][i] if st["wave"] and st["wave"][i] is not None else st["f"]
        if grad:
            p = [D.clone().requires_grad_(), T2.clone().requires_grad_(),
                 torch.tensor(kap, dtype=torch.float64, device=dev, requires_grad=True)]
            M, _ = solver[gi].run(*p, gG, f, grad=True)
            z = M.sum()
            s = z.abs() / M.numel()
            s.backward()
            for n, v in zip(grads, p):
                grads[n].append(v.grad.cpu().numpy())
            S.append(s.item())
            Z.append(z.item())
        else:
            with torch.no_grad():
                M, ser = solver[gi].run(D, T2, kap, gG, f, series=k == "ogse" or case.get("series", False))
            Z.append(M.sum().item())
            S.append(abs(Z[-1]) / M.numel())
            series.append(np.array(ser))
            fields.append(M.reshape(-1) if k in ("tissue", "protocol") or (k == "batch" and gi) else None)
            last = M.reshape(-1)
        del M
    Z = np.array(Z)
    if k == "free":
        return {"Z": Z, "series": np.concatenate(series), "field": last}
    if k in ("plain", "specimen", "links", "slice", "study2d"):
        return {"Z": Z, "field": last}
    if k == "ogse":
        return {"Z": Z, "series": series[0], "field": last}
    if k in ("tissue", "batch", "protocol"):
        return {"Z": Z, "S": np.array(S), "fields": [v for v in fields if v is not None]}
    if k == "gradient":
        return {"Z": Z, "dD": np.array(grads["dD"]), "dT2": np.array(grads["dT2"]), "dkappa": np.array(grads["dkappa"])}
    return {"S": torch.tensor(S[0], dtype=torch.float64), "dD": torch.tensor(grads["dD"][0]),
            "dT2": torch.tensor(grads["dT2"][0]), "dkappa": torch.tensor(grads["dkappa"][0])}
