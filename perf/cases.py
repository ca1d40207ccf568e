"""Performance cases of the membrane dynamics library: what a program that
uses it has it do, through the public calls of the package, from the smallest
patch to the whole red cell.

A case is a dict of plain values; ``kind`` says which call sequence a pass is:

* ``run``     ``System.integrate`` on a membrane that is already set up, then
              its state as CUDA tensors: the production loop between two
              frames of a trajectory;
* ``forces``  ``System.compute_forces`` with the energies, then the forces:
              the monitoring of a run;
* ``setup``   a new membrane from host arrays: handle, particles, bonds,
              k-means cell initialisation, first forces;
* ``quench``  ``System.quench``: the relaxation of a newly built structure;
* ``batch``   a batch of uneven membranes through the arena: admitted
              together, stepped, retired (host arrays in and out).

Membranes are synthetic: flat periodic patches with a honeycomb network,
spherical vesicles and biconcave (Evans-Fung) cells with a triangulated
network, lipids 1.12 sigma apart with 5 % jitter, thermal velocities, all
drawn from the seed on the GPU.  ``exact`` integrates or evaluates the same
membrane in plain FP64 torch, with a neighbour search of its own.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1701_02059_gb300 as G

LIPID, JUNCTION, SPECTRIN, BAND3, GLYCOPHORIN = 0, 1, 2, 3, 4
SPACING = 1.12
PITCH = SPACING * math.sqrt(3.0) / 2.0
AREA = SPACING * PITCH
GOLDEN = math.pi * (3.0 - math.sqrt(5.0))
# Evans-Fung thickness profile (micrometres)
EF_R0, EF_C0, EF_C2, EF_C4 = 3.91, 0.81, 7.83, -4.39
PRECISION = {"f32": G.F32_FORCE_F64_STATE, "f64": G.F64_ALL, "f32step": G.F32_FORCE_F32_STEP}
# species table of the membranes with band-3 and glycophorin (well depth, cutoff)
PROTEIN_EPS = [[0.0, 1.2, 0.9], [1.2, 1.4, 1.1], [0.9, 1.1, 0.0]]
PROTEIN_RC = [[0.0, 2.8, 0.0], [2.8, 2.9, 2.7], [0.0, 2.7, 0.0]]
DEV = "cuda"


def listed():
    return [
        # the smallest system in use: the 2,304-particle patch, periodic in x
        # and y, where a step is launches and latency
        {"name": "patch-2k", "kind": "run", "shape": "patch", "n": 2304, "precision": "f32", "steps": 50},
        # the 62,000-particle vesicle with 20-bead spectrin chains
        {"name": "vesicle-62k", "kind": "run", "shape": "vesicle", "n": 61962, "precision": "f32", "steps": 20},
        # an odd-sized periodic patch at the narrowest precision (FP32 increments)
        {"name": "patch-145k-f32step", "kind": "run", "shape": "patch", "n": 145000, "precision": "f32step", "steps": 10},
        # FP64 pair terms: the reference runs that the FP32 forces are judged by
        {"name": "vesicle-250k-f64", "kind": "run", "shape": "vesicle", "n": 250007, "precision": "f64", "steps": 4},
        # the biconcave cell at about a quarter of its particles
        {"name": "cell-1m", "kind": "run", "shape": "cell", "n": 1000003, "precision": "f32", "steps": 6},
        # with band-3 and glycophorin: species pairs and anchors
        {"name": "cell-1m-proteins", "kind": "run", "shape": "cell", "n": 1000003, "precision": "f32", "steps": 6,
         "proteins": True},
        # cells rebuilt every tenth step, or when a particle has moved 0.3 sigma
        {"name": "cell-1m-skin", "kind": "run", "shape": "cell", "n": 1000003, "precision": "f32", "steps": 20,
         "rebuild_every": 10, "skin": 0.3},
        # the whole red cell, cells rebuilt every step: the main workload
        {"name": "cell-4m", "kind": "run", "shape": "cell", "n": 4000000, "precision": "f32", "steps": 4},
        # energies and forces of the state in hand (monitoring)
        {"name": "forces-1m", "kind": "forces", "shape": "cell", "n": 1000003, "precision": "f32"},
        # a new membrane from host arrays up to its first forces
        {"name": "setup-500k", "kind": "setup", "shape": "vesicle", "n": 500009, "precision": "f32"},
        # relaxation of a new structure: forces and rebuild every step, no noise
        {"name": "quench-62k", "kind": "quench", "shape": "vesicle", "n": 61962, "precision": "f32", "steps": 10},
        # uneven patches and vesicles in one batch (an ensemble, a served stream)
        {"name": "batch-12", "kind": "batch", "n": 100000, "count": 12, "precision": "f32", "steps": 80},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "forces", "setup", "quench", "batch"])
    if kind == "batch":
        return {"kind": "batch", "n": _log_uniform(rng, 8_000, 100_000), "count": rng.randint(3, 12), "precision": "f32",
                "steps": rng.randint(20, 80)}
    precision = rng.choice(["f32", "f32", "f32", "f32step", "f64"])
    # (a cell needs about 400,000 particles for its network's straight chains
    # to follow the surface)
    shape = rng.choice(["patch", "vesicle"] if precision == "f64" else ["patch", "vesicle", "cell"])
    hi = {"run": 2_000_000, "forces": 2_000_000, "setup": 500_000, "quench": 500_000}[kind]
    if precision == "f64":
        hi = min(hi, 200_000)
    case = {"kind": kind, "shape": shape, "n": _log_uniform(rng, 400_000 if shape == "cell" else 2_304, hi),
            "precision": precision}
    if kind in ("run", "quench"):
        case["steps"] = rng.randint(2, 8) if case["n"] > 200_000 else rng.randint(4, 20)
    if kind in ("run", "forces") and precision != "f64":
        option = rng.choice(["", "", "proteins", "skin"])
        if option == "proteins" and shape == "cell":
            case["proteins"] = True
        elif option == "skin" and kind == "run":
            case["rebuild_every"] = rng.randint(4, 12)
            case["skin"] = round(rng.uniform(0.2, 0.4), 3)
    return case


# ------------------------------------------------------------------ membranes
def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, dtype=torch.float64, device=DEV)


def _icosphere(f):
    """Unit icosphere of frequency f: vertices [10 f^2 + 2, 3] and its edges."""
    p = (1.0 + math.sqrt(5.0)) / 2.0
    v0 = np.array([[-1, p, 0], [1, p, 0], [-1, -p, 0], [1, -p, 0], [0, -1, p], [0, 1, p], [0, -1, -p], [0, 1, -p],
                   [p, 0, -1], [p, 0, 1], [-p, 0, -1], [-p, 0, 1]])
    side = np.linalg.norm(v0[:, None] - v0[None], axis=2) < 2.01
    faces = [(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
             if side[a, b] and side[b, c] and side[a, c]]
    i, j = np.meshgrid(np.arange(f + 1), np.arange(f + 1), indexing="ij")
    keep = i + j <= f
    ij = np.stack([i[keep], j[keep]], 1)
    at = -np.ones((f + 2, f + 2), np.int64)
    at[ij[:, 0], ij[:, 1]] = np.arange(len(ij))
    e = []
    for di, dj in ((1, 0), (0, 1), (1, -1)):
        q = ij + [di, dj]
        ok = (q.min(1) >= 0) & (q.sum(1) <= f)
        e.append(np.stack([at[ij[ok, 0], ij[ok, 1]], at[q[ok, 0], q[ok, 1]]], 1))
    e = np.concatenate(e)
    w = np.concatenate([ij, f - ij.sum(1, keepdims=True)], 1) / f
    pts = np.concatenate([w @ v0[list(t)] for t in faces])
    pts /= np.linalg.norm(pts, axis=1, keepdims=True)
    edges = np.concatenate([e + k * len(ij) for k in range(len(faces))])
    key = np.round(pts * 1e7).astype(np.int64)
    _, first, inv = np.unique(key, axis=0, return_index=True, return_inverse=True)
    edges = np.unique(np.sort(inv.reshape(-1)[edges], 1), axis=0)
    return pts[first], edges


def _meridian(t):
    s, c = torch.sin(t), torch.cos(t)
    s2 = s * s
    prof = EF_C0 + EF_C2 * s2 + EF_C4 * s2 * s2
    dprof = (EF_C2 + 2.0 * EF_C4 * s2) * 2.0 * s * c
    return EF_R0 * s, 0.5 * c * prof, EF_R0 * c, 0.5 * (-s * prof + c * dprof)


def _cell_table():
    # (on the host: a running sum on the GPU may differ between two runs)
    t = torch.linspace(0.0, math.pi, 200001, dtype=torch.float64)
    r, _, dr, dz = _meridian(t)
    da = 2.0 * math.pi * r * torch.sqrt(dr * dr + dz * dz)
    area = torch.cat([t.new_zeros(1), torch.cumsum(0.5 * (da[1:] + da[:-1]) * (t[1] - t[0]), 0)])
    return t.to(DEV), area.to(DEV)


def _surface(unit, shape, area_total):
    """Points and outward normals on the sphere or the biconcave cell of the
    given area for points of the unit sphere (equal areas map to equal areas)."""
    if shape == "vesicle":
        return unit * math.sqrt(area_total / (4.0 * math.pi)), unit
    t, area = _cell_table()
    u = ((1.0 - unit[:, 2]) * 0.5).clamp(0.0, 1.0) * area[-1]
    k = torch.searchsorted(area, u).clamp(1, len(area) - 1)
    f = (u - area[k - 1]) / (area[k] - area[k - 1])
    r, z, dr, dz = _meridian(t[k - 1] + f * (t[k] - t[k - 1]))
    m = torch.sqrt(dr * dr + dz * dz)
    phi = torch.atan2(unit[:, 1], unit[:, 0])
    cp, sp = torch.cos(phi), torch.sin(phi)
    scale = math.sqrt(area_total / float(area[-1]))
    return (torch.stack([r * cp, r * sp, z], 1) * scale,
            torch.stack([-dz / m * cp, -dz / m * sp, dr / m], 1))


def _closed(shape, n, gen):
    """Closed membrane of about n particles: Fibonacci lipids and a network
    1 sigma inside (20-bead chains in a vesicle, 4-bead chains in a cell)."""
    beads = 20 if shape == "vesicle" else 4
    per_junction = 3 * beads + 1
    lipids_per_junction = 110.0
    f = max(1, round(math.sqrt(n / (lipids_per_junction + per_junction) / 10.0)))
    nj, ne = 10 * f * f + 2, 30 * f * f
    nl = max(n - nj - ne * beads, 1000)
    area = nl * AREA
    k = torch.arange(nl, dtype=torch.float64, device=DEV)
    z = 1.0 - (2.0 * k + 1.0) / nl
    s = torch.sqrt((1.0 - z * z).clamp(min=0.0))
    lp, lo = _surface(torch.stack([s * torch.cos(k * GOLDEN), s * torch.sin(k * GOLDEN), z], 1), shape, area)
    noise = 0.05 * _normal(gen, nl, 3)
    lp = lp + noise - (noise * lo).sum(1, keepdim=True) * lo
    if shape == "vesicle":
        lo = lp / lp.norm(dim=1, keepdim=True)
    vj, edges = _icosphere(f)
    vj = torch.from_numpy(vj).to(DEV)
    jp, jn = _surface(vj, shape, area)
    jp = jp - jn
    e = torch.from_numpy(edges).to(DEV)
    a, d = jp[e[:, 0]], jp[e[:, 1]] - jp[e[:, 0]]
    w = torch.arange(1, beads + 1, dtype=torch.float64, device=DEV) / (beads + 1)
    bp = (a[:, None] + d[:, None] * w[None, :, None]).reshape(-1, 3)
    if shape == "vesicle":
        bp = bp * (math.sqrt(area / (4.0 * math.pi)) - 1.0) / bp.norm(dim=1, keepdim=True)
    r0 = (1.03 * d.norm(dim=1) / (beads + 1)).repeat_interleave(beads + 1)
    return lp, lo, jp, bp, e, r0, [0.0, 0.0, 0.0], [0, 0, 0], 61.0


def _patch(n, gen):
    """Flat patch periodic in x and y: 576 m^2 particles, honeycomb network of
    10-bead chains 1 sigma below."""
    m = max(2, round(math.sqrt(n / 576.0)))
    nx, ny, beads = 16 * m, 32 * m, 10
    lx, ly = nx * SPACING, ny * PITCH
    j, i = torch.meshgrid(torch.arange(ny, device=DEV), torch.arange(nx, device=DEV), indexing="ij")
    lp = torch.stack([i * SPACING + (j % 2) * (SPACING / 2), j * PITCH, torch.zeros_like(i)], -1).reshape(-1, 3).double()
    lp[:, :2] += 0.05 * _normal(gen, nx * ny, 2)
    lo = torch.cat([math.radians(5.0) * _normal(gen, nx * ny, 2), torch.ones(nx * ny, 1, dtype=torch.float64, device=DEV)], 1)
    lo = lo / lo.norm(dim=1, keepdim=True)
    b = lx / (m * math.sqrt(3.0))
    base = np.array([[0.0, 0.0], [0.0, b], [math.sqrt(3.0) / 2 * b, 1.5 * b], [math.sqrt(3.0) / 2 * b, 2.5 * b]])
    ux, uy = (q.reshape(-1) for q in np.meshgrid(np.arange(m), np.arange(m), indexing="ij"))
    xy = (base[None] + np.stack([ux * math.sqrt(3.0) * b, uy * 3.0 * b], 1)[:, None]).reshape(-1, 2)
    vid = lambda x, y, s: ((x % m) * m + y % m) * 4 + s  # noqa: E731
    e = np.concatenate([np.stack([vid(ux, uy, s), vid(ux + dx, uy + dy, t)], 1) for s, t, dx, dy in
                        ((0, 1, 0, 0), (1, 2, 0, 0), (2, 3, 0, 0), (3, 0, 0, 1), (1, 2, -1, 0), (3, 0, 1, 1))])
    jp = np.concatenate([(xy + [0.25 * SPACING, 0.25 * PITCH]) % [lx, ly], np.full((len(xy), 1), -1.0)], 1)
    jp, e = torch.from_numpy(jp).to(DEV), torch.from_numpy(e).to(DEV)
    box = torch.tensor([lx, ly], dtype=torch.float64, device=DEV)
    d = jp[e[:, 1]] - jp[e[:, 0]]
    d[:, :2] -= box * torch.round(d[:, :2] / box)
    w = torch.arange(1, beads + 1, dtype=torch.float64, device=DEV) / (beads + 1)
    bp = (jp[e[:, 0]][:, None] + d[:, None] * w[None, :, None]).reshape(-1, 3)
    bp[:, :2] = torch.remainder(bp[:, :2], box)
    r0 = torch.ones(len(e) * (beads + 1), dtype=torch.float64, device=DEV)
    return lp, lo, jp, bp, e, r0, [lx, ly, 0.0], [1, 1, 0], 36.0


def _membrane(shape, n, seed, proteins=False, kT=0.2):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 2 + 1)
    lp, lo, jp, bp, e, r0, box, periodic, per_cell = _patch(n, gen) if shape == "patch" else _closed(shape, n, gen)
    nl, nj, ne = len(lp), len(jp), len(e)
    beads = len(bp) // ne
    chain = nl + nj + torch.arange(ne * beads, device=DEV).reshape(ne, beads)
    path = torch.cat([nl + e[:, :1], chain, nl + e[:, 1:]], 1)
    bonds = torch.stack([path[:, :-1], path[:, 1:]], 2).reshape(-1, 2)
    kb = torch.full_like(r0, 100.0)
    pos = torch.cat([lp, jp, bp])
    ori = torch.zeros_like(pos)
    ori[:nl] = lo
    typ = torch.full((len(pos),), SPECTRIN, dtype=torch.uint8, device=DEV)
    typ[:nl] = LIPID
    typ[nl:nl + nj] = JUNCTION
    if proteins:
        # a glycophorin over every junction and a band-3 over a quarter of the
        # beads (the nearest lipid each, anchored to it), 5 % of the other
        # lipids as mobile band-3
        pick = nl + nj + torch.randperm(len(bp), generator=gen, device=DEV)[:len(bp) // 4]
        want = torch.cat([torch.arange(nl, nl + nj, device=DEV), pick])
        mine = torch.zeros(len(pos), dtype=torch.bool, device=DEV)
        mine[want] = True
        i, j = _close_pairs(pos, 2.0, box, periodic)
        i, j = torch.cat([i, j]), torch.cat([j, i])
        ok = mine[i] & (j < nl)
        i, j = i[ok], j[ok]
        d = (pos[i] - pos[j]).norm(dim=1)
        order = torch.argsort(d, stable=True)
        first = torch.full((len(pos),), len(order), device=DEV)
        first.scatter_reduce_(0, i[order], torch.arange(len(order), device=DEV), "amin")
        got = want[first[want] < len(order)]
        lip = j[order][first[got]]
        owner = torch.full((nl,), len(pos), device=DEV)
        owner.scatter_reduce_(0, lip, got, "amin")
        keep = owner[lip] == got
        got, lip = got[keep], lip[keep]
        free = torch.ones(nl, dtype=torch.bool, device=DEV)
        free[lip] = False
        rest = free.nonzero()[:, 0]
        typ[rest[torch.randperm(len(rest), generator=gen, device=DEV)[:len(rest) // 20]]] = BAND3
        typ[lip] = torch.where(got < nl + nj, GLYCOPHORIN, BAND3).to(torch.uint8)
        bonds = torch.cat([bonds, torch.stack([lip, got], 1)])
        r0 = torch.cat([r0, (pos[lip] - pos[got]).norm(dim=1)])
        kb = torch.cat([kb, torch.full((len(lip),), 50.0, dtype=torch.float64, device=DEV)])
    bil = (typ == LIPID) | (typ >= BAND3)
    vel = math.sqrt(kT) * _normal(gen, len(pos), 3)
    w = math.sqrt(kT) * _normal(gen, len(pos), 3)
    w = (w - (w * ori).sum(1, keepdim=True) * ori) * bil[:, None]
    host = lambda t, d: np.ascontiguousarray(t.cpu().numpy().astype(d, copy=False))  # noqa: E731
    return SimpleNamespace(pos=host(pos, np.float64), vel=host(vel, np.float64), ori=host(ori, np.float64),
                           angvel=host(w, np.float64), type=host(typ, np.uint8),
                           id=np.arange(len(pos), dtype=np.uint32), bonds=host(bonds, np.int32),
                           r0=host(r0, np.float64), kb=host(kb, np.float64), box=box, periodic=periodic, kT=kT,
                           n=len(pos), n_centroids=max(1, round(len(pos) / per_cell)), proteins=bool(proteins))


def _params(case, mem, seed):
    kw = {}
    if mem.proteins:
        kw.update(eps_mem=PROTEIN_EPS, rc_mem=PROTEIN_RC)
    if case.get("skin"):
        kw.update(rebuild_every=case["rebuild_every"], skin=case["skin"])
    return G.make_params(kT=mem.kT, n_centroids=mem.n_centroids, box=mem.box, periodic=mem.periodic, seed=int(seed),
                         precision=PRECISION[case["precision"]], **kw)


def _batch_members(case, seed):
    """Sizes of a batch: patches and vesicles in turn, evenly spread in the
    logarithm from 5,000 particles up, temperatures 0.1 to 0.3."""
    c = case["count"]
    for k in range(c):
        n = int(5000 * (case["n"] / 5000.0) ** (k / max(c - 1, 1)))
        yield "patch" if k % 2 else "vesicle", n, seed * 64 + k, 0.1 + 0.2 * k / max(c - 1, 1)


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    if case["kind"] == "batch":
        mems = [_membrane(s, n, q, kT=kT) for s, n, q, kT in _batch_members(case, seed)]
        for m in mems:
            m.n_centroids = max(1, round(m.n / 61))
        arena = G.Arena(64 << 30, PRECISION[case["precision"]])
        return SimpleNamespace(case=case, arena=arena,
                               items=[(_params(case, m, seed * 64 + k), m, case["steps"]) for k, m in enumerate(mems)])
    mem = _membrane(case["shape"], case["n"], seed, case.get("proteins", False))
    if case["kind"] == "setup":
        return SimpleNamespace(case=case, mem=mem, params=_params(case, mem, seed))
    system = G.System(_params(case, mem, seed))
    system.load_membrane(mem)
    system.init_cells()
    return SimpleNamespace(case=case, system=system)


def run(state):
    case = state.case
    if case["kind"] == "run":
        state.system.integrate(case["steps"])
        return state.system.state_tensors()
    if case["kind"] == "forces":
        energies = state.system.compute_forces(energies=True)
        force, torque = state.system.force_tensors()
        return {"energies": energies, "force": force, "torque": torque}
    if case["kind"] == "quench":
        fmax = state.system.quench(case["steps"], 0.005)
        out = state.system.state_tensors()
        return {"fmax": fmax, "pos": out["pos"], "ori": out["ori"]}
    if case["kind"] == "setup":
        with G.System(state.params) as system:
            system.load_membrane(state.mem)
            system.init_cells()
            system.compute_forces()
            force, torque = system.force_tensors()
            cells = system.cells()
        del cells["adj"]   # its length depends on the membrane; adj_ptr holds the row lengths
        return {"force": force, "torque": torque, "cells": cells}
    slots = state.arena.admit_many(state.items)
    left = set(slots)
    done = {}
    while left:
        state.arena.run(case["steps"])
        for s in state.arena.poll():
            done[s] = state.arena.retire(s)
            left.discard(s)
    return [done[s] for s in slots]


def _counts(case):
    """(particles, bilayer particles, bonds) of a case's membrane, about."""
    if case["kind"] == "batch":
        sizes = [(n, s) for s, n, _, _ in _batch_members(case, 0)]
    else:
        sizes = [(case["n"], case["shape"])]
    share = {"patch": 0.89, "vesicle": 0.65, "cell": 0.89}
    return (sum(n for n, _ in sizes), sum(n * share[s] for n, s in sizes), sum(n * (1.0 - share[s]) for n, s in sizes))


def work(case):
    """The state in and out once per step (x, v of every particle, n, w of the
    bilayer's, 8 bytes a component); per step about 10 pairs per bilayer
    particle (100 operations a pair and half as many again for the second
    side) and 200 operations per particle of the integrator."""
    n, nb, bonds = _counts(case)
    pair_flops = 10.0 * nb * 150.0 + 30.0 * bonds
    state = 48.0 * n + 48.0 * nb
    if case["kind"] in ("run", "quench", "batch"):
        steps = case["steps"]
        return {"bytes": 2.0 * state * steps, "flops": (pair_flops + 200.0 * n) * steps}
    if case["kind"] == "forces":
        return {"bytes": 24.0 * n + 24.0 * nb + 48.0 * n, "flops": pair_flops}
    # set-up: the host arrays in; the forces, cells and storage order out;
    # ten rounds of assignment over about ten candidates each
    return {"bytes": 101.0 * n + 56.0 * n, "flops": pair_flops + 10.0 * 10.0 * 9.0 * n}


# ------------------------------------------------------------------ FP64 reference
def _close_pairs(x, rc, box, periodic):
    """All pairs (i, j), each once, closer than rc: particles binned on a grid
    of edge >= rc, every bin against itself and half of its 26 neighbours."""
    lo = x.min(0).values
    dims, rel = [], []
    for a in range(3):
        if periodic[a]:
            d = max(3, int(box[a] / rc))
            g = torch.floor(torch.remainder(x[:, a], box[a]) * (d / box[a])).long().clamp(0, d - 1)
        else:
            g = torch.floor((x[:, a] - lo[a]) / rc).long() + 1
            d = int(g.max()) + 2
        dims.append(d)
        rel.append(g)
    gx, gy, gz = rel
    key = (gz * dims[1] + gy) * dims[0] + gx
    order = torch.argsort(key, stable=True)
    ks = key[order]
    uniq, cnt = torch.unique_consecutive(ks, return_counts=True)
    start = torch.cumsum(cnt, 0) - cnt
    rank = torch.empty_like(order)
    rank[order] = torch.arange(len(order), device=x.device)
    out_i, out_j = [], []
    offsets = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1) if (dz, dy, dx) >= (0, 0, 0)]
    bx = torch.tensor([b if p else 1.0 for b, p in zip(box, periodic)], dtype=x.dtype, device=x.device)
    per = torch.tensor([float(p) for p in periodic], dtype=x.dtype, device=x.device)
    for dx, dy, dz in offsets:
        q = []
        for g, d, a in ((gx, dx, 0), (gy, dy, 1), (gz, dz, 2)):
            h = g + d
            q.append(torch.remainder(h, dims[a]) if periodic[a] else h)
        k2 = (q[2] * dims[1] + q[1]) * dims[0] + q[0]
        b = torch.searchsorted(uniq, k2).clamp(max=len(uniq) - 1)
        m = torch.where(uniq[b] == k2, cnt[b], torch.zeros_like(b))
        i = torch.repeat_interleave(torch.arange(len(x), device=x.device), m)
        first = torch.repeat_interleave(start[b], m)
        base = torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        j = order[first + torch.arange(len(i), device=x.device) - base]
        if (dx, dy, dz) == (0, 0, 0):
            ok = rank[i] < rank[j]
            i, j = i[ok], j[ok]
        d = x[j] - x[i]
        d = d - per * bx * torch.round(d / bx)
        ok = (d * d).sum(1) < rc * rc
        out_i.append(i[ok])
        out_j.append(j[ok])
    return torch.cat(out_i), torch.cat(out_j)


class _Exact:
    """The model's forces and BAOAB steps in FP64 torch."""

    def __init__(self, mem, seed):
        put = lambda a, d: torch.from_numpy(np.ascontiguousarray(a)).to(DEV).to(d)  # noqa: E731
        f = torch.float64
        self.x, self.v, self.n, self.w = (put(a, f) for a in (mem.pos, mem.vel, mem.ori, mem.angvel))
        typ = put(mem.type, torch.int64)
        self.bil = (typ == LIPID) | (typ >= BAND3)
        self.species = torch.where(typ >= BAND3, typ - 2, torch.zeros_like(typ))
        self.bonds, self.r0, self.kb = put(mem.bonds, torch.int64), put(mem.r0, f), put(mem.kb, f)
        self.box = torch.tensor([b if p else 1.0 for b, p in zip(mem.box, mem.periodic)], dtype=f, device=DEV)
        self.per = torch.tensor([float(p) for p in mem.periodic], dtype=f, device=DEV)
        self.mem, self.seed, self.kT = mem, int(seed), mem.kT
        eps, rc = np.array(PROTEIN_EPS if mem.proteins else np.zeros((3, 3))), np.array(
            PROTEIN_RC if mem.proteins else np.zeros((3, 3)))
        self.eps = torch.from_numpy(np.where(eps > 0, eps, 1.0)).to(DEV)
        self.rc = torch.from_numpy(np.where(rc > 0, rc, 2.6)).to(DEV)
        # pairs bonded to each other or to a common partner carry no WCA term
        n = len(self.x)
        a, b = torch.cat([self.bonds[:, 0], self.bonds[:, 1]]), torch.cat([self.bonds[:, 1], self.bonds[:, 0]])
        o = torch.argsort(a)
        a, b = a[o], b[o]
        cnt = torch.bincount(a, minlength=n)
        st = torch.cumsum(cnt, 0) - cnt
        m = cnt[b]
        src = torch.repeat_interleave(a, m)
        off = torch.arange(len(src), device=DEV) - torch.repeat_interleave(torch.cumsum(m, 0) - m, m)
        far = b[torch.repeat_interleave(st[b], m) + off]
        lo = torch.cat([torch.minimum(a, b), torch.minimum(src, far)])
        hi = torch.cat([torch.maximum(a, b), torch.maximum(src, far)])
        self.excluded = torch.unique(lo * n + hi)

    def _image(self, d):
        return d - self.per * self.box * torch.round(d / self.box)

    def forces(self):
        """Forces, torques and [U_pair, U_bond, K_trans, K_rot, W]."""
        x, n = self.x, self.n
        rmin, zeta, mu = 2.0 ** (1.0 / 6.0), 4, 3.0
        F, T = torch.zeros_like(x), torch.zeros_like(x)
        i, j = _close_pairs(x, float(self.rc.max()), self.mem.box, self.mem.periodic)
        d = self._image(x[i] - x[j])
        r = d.norm(dim=1)
        both = self.bil[i] & self.bil[j]
        s = self.species
        ll = both & (r < self.rc[s[i], s[j]])
        u_pair = virial = 0.0
        # bilayer pairs
        a, b, dd, rr = i[ll], j[ll], d[ll], r[ll]
        eps, rc = self.eps[s[a], s[b]], self.rc[s[a], s[b]]
        h, na, nb = dd / rr[:, None], n[a], n[b]
        nar, nbr = (na * h).sum(1), (nb * h).sum(1)
        phi = 1.0 + mu * ((na * nb).sum(1) - nar * nbr - 1.0)
        near = rr < rmin
        q2 = (rmin / rr) ** 2
        th = 0.5 * math.pi * (rr - rmin) / (rc - rmin)
        c, sn = torch.cos(th), torch.sin(th)
        f = torch.where(near, eps * (q2 * q2 - 2.0 * q2) + eps, torch.zeros_like(rr))
        fp = torch.where(near, 4.0 * eps * (q2 - q2 * q2) / rr, torch.zeros_like(rr))
        g = torch.where(near, -eps, -eps * c ** (2 * zeta))
        gp = torch.where(near, torch.zeros_like(rr), eps * 2 * zeta * c ** (2 * zeta - 1) * sn * 0.5 * math.pi / (rc - rmin))
        u_pair += float((f + g * phi).sum())
        w = -nbr[:, None] * na - nar[:, None] * nb
        gm = (g * mu)[:, None]
        fv = -(fp + gp * phi)[:, None] * h - gm * (w - (w * h).sum(1, keepdim=True) * h) / rr[:, None]
        F.index_add_(0, a, fv)
        F.index_add_(0, b, -fv)
        T.index_add_(0, a, -gm * torch.linalg.cross(na, nb - nbr[:, None] * h))
        T.index_add_(0, b, -gm * torch.linalg.cross(nb, na - nar[:, None] * h))
        virial += float((dd * fv).sum())
        # excluded volume of the cytoskeleton
        sig = torch.where(self.bil[i] | self.bil[j], 1.0, 0.5).double()
        wca = ~both & (r < rmin * sig)
        a, b, dd, rr, sig = i[wca], j[wca], d[wca], r[wca], sig[wca]
        key = torch.minimum(a, b) * len(x) + torch.maximum(a, b)
        at = torch.searchsorted(self.excluded, key).clamp(max=len(self.excluded) - 1)
        ok = self.excluded[at] != key
        a, b, dd, rr, sig = a[ok], b[ok], dd[ok], rr[ok], sig[ok]
        s6 = (sig / rr) ** 6
        u_pair += float((4.0 * (s6 * s6 - s6) + 1.0).sum())
        fv = (4.0 * (12.0 * s6 * s6 - 6.0 * s6) / (rr * rr))[:, None] * dd
        F.index_add_(0, a, fv)
        F.index_add_(0, b, -fv)
        virial += float((dd * fv).sum())
        # bonds
        a, b = self.bonds[:, 0], self.bonds[:, 1]
        dd = self._image(x[a] - x[b])
        rr = dd.norm(dim=1)
        fv = (-self.kb * (rr - self.r0) / rr)[:, None] * dd
        F.index_add_(0, a, fv)
        F.index_add_(0, b, -fv)
        virial += float((dd * fv).sum())
        u_bond = float((0.5 * self.kb * (rr - self.r0) ** 2).sum())
        k_rot = float(0.5 * (self.w[self.bil] ** 2).sum())
        return F, T, [u_pair, u_bond, float(0.5 * (self.v ** 2).sum()), k_rot, virial]

    def _philox(self, step, sub):
        mask = 0xFFFFFFFF

        def mul(m, c):
            lo = m * (c & 0xFFFF)
            s = (lo >> 16) + m * (c >> 16)
            return s >> 16, ((s & 0xFFFF) << 16) | (lo & 0xFFFF)

        c0 = torch.arange(len(self.x), device=DEV)
        c1, c2, c3 = (torch.full_like(c0, q) for q in (step & mask, step >> 32, sub))
        k0, k1 = self.seed & mask, (self.seed >> 32) & mask
        for _ in range(10):
            h0, l0 = mul(0xD2511F53, c0)
            h1, l1 = mul(0xCD9E8D57, c2)
            c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        u = (torch.stack([c0, c1, c2], 1).double() + 0.5) / 4294967296.0 - 0.5
        return math.sqrt(12.0) * u

    def _turn(self, h):
        a = 0.5 * h * self.w
        b = torch.linalg.cross(a, self.n)
        self.n = self.n + 2.0 / (1.0 + (a * a).sum(1, keepdim=True)) * (b + torch.linalg.cross(a, b))

    def _kick(self, h, F, T):
        self.v = self.v + h * F
        self.w = self.w + h * (T - (T * self.n).sum(1, keepdim=True) * self.n) * self.bil[:, None]

    def integrate(self, steps, dt=0.01):
        F, T, _ = self.forces()
        h, e = 0.5 * dt, math.exp(-dt)
        s = math.sqrt((1.0 - e * e) * self.kT)
        for k in range(steps):
            self._kick(h, F, T)
            self.x = self.x + h * self.v
            self._turn(h)
            self.v = e * self.v + s * self._philox(k, 0)
            z = self._philox(k, 1)
            z = (z - (z * self.n).sum(1, keepdim=True) * self.n) * self.bil[:, None]
            self.w = e * self.w + s * z
            self.x = self.x + h * self.v
            self._turn(h)
            self.n = self.n / self.n.norm(dim=1, keepdim=True).clamp(min=1e-300) * self.bil[:, None]
            F, T, _ = self.forces()
            self._kick(h, F, T)
        return {"pos": self.x, "vel": self.v, "ori": self.n, "angvel": self.w}

    def quench(self, steps, dt, max_move=0.02, max_turn=0.05):
        def follow(u, f, limit):
            uf, ff = (u * f).sum(1, keepdim=True), (f * f).sum(1, keepdim=True)
            u = torch.where((uf > 0) & (ff > 0), uf / ff.clamp(min=1e-300) * f, torch.zeros_like(u))
            m = dt * u.norm(dim=1, keepdim=True)
            return torch.where(m > limit, u * (limit / m.clamp(min=1e-300)), u)

        F, T, _ = self.forces()
        for _ in range(steps):
            self.v = follow(self.v + dt * F, F, max_move)
            t = (T - (T * self.n).sum(1, keepdim=True) * self.n) * self.bil[:, None]
            self.w = follow(self.w + dt * t, t, max_turn)
            self.x = self.x + dt * self.v
            self._turn(dt)
            self.n = self.n / self.n.norm(dim=1, keepdim=True).clamp(min=1e-300) * self.bil[:, None]
            F, T, _ = self.forces()
        return {"fmax": float(F.norm(dim=1).max()), "pos": self.x, "ori": self.n}


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for k, (shape, n, q, kT) in enumerate(_batch_members(case, seed)):
            e = _Exact(_membrane(shape, n, q, kT=kT), seed * 64 + k)
            out.append({key: v.cpu().numpy() for key, v in e.integrate(case["steps"]).items()} | {"step": None})
        return out
    e = _Exact(_membrane(case["shape"], case["n"], seed, case.get("proteins", False)), seed)
    if case["kind"] == "run":
        return e.integrate(case["steps"])
    if case["kind"] == "quench":
        return e.quench(case["steps"], 0.005)
    F, T, energies = e.forces()
    if case["kind"] == "forces":
        return {"energies": np.array(energies), "force": F, "torque": T}
    # the cells are decided by comparisons and integers, which have to be equal
    return {"force": F, "torque": T, "cells": None}
