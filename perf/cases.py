"""What is measured: the work that programs built on this library ask of it.

Every case is one pass through the public Python binding, on inputs made from
a seed alone.  The kinds:

  step      a resident simulation advances by some steps and its state is
            read back on the device (the md_step loop of a long run): the
            mixed form, the FP64 form and the cell-list-only variant
  load      a configuration is loaded, measured and its forces read: one-shot
            evaluation of many configurations through one handle
  ensemble  resident replicas of uneven size advance in one launch and are
            read back
  batch     requests are admitted, run and retired: what the serving loop does
            with each of its requests
  noalloc   forces, energy and virial of one configuration in the fixed
            scratch area

Inputs are melted fluids.  A periodic tile of at most 2048 atoms is taken from
a jittered FCC lattice and run forward with plain torch (all pairs, FP32) for
some hundred steps, then repeated over the box; velocities are drawn for every
atom.  So a state of any size has the pair distances of the fluid and depends
on nothing but the seed.

Positions are returned as displacements over the pass (minimum image), so that
an atom that crosses the periodic boundary one rounding earlier or later does
not look like an error of a box length.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_0911_5631_gb300 as md

RC = md.WCA_RC
DT = 0.005
TILE = 2048          # most atoms of the melted tile
MELT = 300           # steps of its melt


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The smallest system of the test and benchmark configurations that is
        # advanced by neighbour list: launches and their gaps are the cost.
        dict(name="step_2k", kind="step", n=2048, rho=0.8, T=1.0, rc=RC, skin=0.4, form="mixed", cells=False,
             steps=100),
        # A middling system of odd size in a box that is no cube (requests of
        # the serving configuration run from 500 to 200000 atoms).
        dict(name="step_20k_odd", kind="step", n=20011, rho=0.7, T=1.5, rc=RC, skin=0.4, form="mixed", cells=False,
             steps=100, ay=1.3, az=0.8),
        # The headline: 1M soft spheres, mixed precision.
        dict(name="step_1m", kind="step", n=1048576, rho=0.8, T=1.0, rc=RC, skin=0.4, form="mixed", cells=False,
             steps=100),
        # The largest configuration, dense and hot.
        dict(name="step_8m", kind="step", n=8388608, rho=1.0, T=2.0, rc=RC, skin=0.4, form="mixed", cells=False,
             steps=20),
        # The FP64 form at the headline size: reference runs.
        dict(name="fp64_1m", kind="step", n=1048576, rho=0.8, T=1.0, rc=RC, skin=0.4, form="fp64", cells=False,
             steps=20),
        # Cell list only, FP64, 2048 atoms: the small parity configuration.
        dict(name="cells_fp64_2k", kind="step", n=2048, rho=0.8, T=1.0, rc=RC, skin=0.0, form="fp64", cells=True,
             steps=50),
        # The Lennard-Jones system of the paper's comparisons.
        dict(name="lj_1m", kind="step", n=1048576, rho=0.38, T=1.2, rc=3.0, skin=0.8, form="mixed", cells=False,
             steps=20),
        # One-shot evaluation of configurations that a program keeps on the
        # device (training data, snapshots): load, energies, forces.
        dict(name="load_100k", kind="load", n=100003, rho=0.8, T=1.0, rc=RC, skin=0.4, form="mixed"),
        # Replicas of the batched-ensemble configuration, resident, between
        # two read-backs.
        dict(name="ensemble_160", kind="ensemble", replicas=160, n_min=256, n_max=32768, steps=100),
        # The serving loop's calls for a batch of requests: admit, run, read
        # back, free.
        dict(name="batch_32", kind="batch", replicas=32, n_min=500, n_max=16000, steps=100),
        # Forces without allocation: a small molecule-sized box, and the
        # largest size that the scratch area takes.
        dict(name="noalloc_500", kind="noalloc", n=500, rho=0.8, rc=RC),
        dict(name="noalloc_64k", kind="noalloc", n=65000, rho=0.8, rc=RC),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "fp64", "cells", "lj", "load", "ensemble", "batch", "noalloc"])
    rho, T = round(rng.uniform(0.6, 1.0), 3), round(rng.uniform(0.5, 2.0), 3)
    if kind in ("step", "fp64"):
        c = dict(kind="step", n=_log_int(rng, 500, 4000000 if kind == "step" else 600000), rho=rho, T=T, rc=RC,
                 skin=rng.choice([0.3, 0.4, 0.4, 0.6]), form="mixed" if kind == "step" else "fp64", cells=False,
                 steps=20)
        if rng.random() < 0.4:  # a box that is no cube
            c["ay"], c["az"] = round(rng.uniform(0.8, 1.5), 2), round(rng.uniform(0.8, 1.5), 2)
        return c
    if kind == "cells":
        form = rng.choice(["mixed", "fp64"])
        return dict(kind="step", n=_log_int(rng, 500, 300000 if form == "mixed" else 100000), rho=rho, T=T, rc=RC,
                    skin=0.0, form=form, cells=True, steps=20)
    if kind == "lj":
        return dict(kind="step", n=_log_int(rng, 5000, 600000), rho=round(rng.uniform(0.3, 0.5), 3), T=1.2,
                    rc=rng.choice([2.2, 2.5, 3.0]), skin=rng.choice([0.4, 0.8]), form="mixed", cells=False, steps=20)
    if kind == "load":
        return dict(kind="load", n=_log_int(rng, 500, 400000), rho=rho, T=T, rc=RC, skin=0.4,
                    form=rng.choice(["mixed", "mixed", "fp64"]))
    if kind == "ensemble":
        return dict(kind="ensemble", replicas=_log_int(rng, 8, 160), n_min=256, n_max=_log_int(rng, 2048, 32768),
                    steps=50)
    if kind == "batch":
        return dict(kind="batch", replicas=_log_int(rng, 1, 48), n_min=500, n_max=_log_int(rng, 1000, 32000), steps=50)
    # (the scratch area holds 65536 cells of width r_c too)
    return dict(kind="noalloc", n=_log_int(rng, 200, min(65000, int(88000 * rho))), rho=rho, rc=RC)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _fcc(n, L):
    """n sites of an FCC lattice that fills the box, spread evenly over it."""
    a0 = (4.0 * float(np.prod(L)) / n) ** (1.0 / 3.0)
    k = np.maximum(1, np.round(L / a0)).astype(int)
    while 4 * int(np.prod(k)) < n:
        k[np.argmin(k * a0 / L)] += 1
    basis = np.array([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]])
    g = np.stack(np.meshgrid(*[np.arange(m) for m in k], indexing="ij"), -1).reshape(-1, 1, 3)
    sites = ((g + 0.25 + basis[None]) * (L / k)).reshape(-1, 3) - 0.5 * L
    return sites[(np.arange(n) * len(sites)) // n]


def _melt(n, L, T, rc, gen):
    """Positions of n[b] atoms in the periodic box L[b] after MELT steps from
    a jittered lattice, the velocities rescaled to T[b] every 20 steps; the
    systems are run side by side, padded to the longest."""
    dev = _dev()
    m = max(n)
    Lt = torch.tensor(np.array(L), dtype=torch.float32, device=dev)[:, None, None, :]
    Tt = torch.tensor(T, dtype=torch.float32, device=dev)
    nt = torch.tensor(n, dtype=torch.float32, device=dev)
    real = torch.arange(m, device=dev)[None, :] < torch.tensor(n, device=dev)[:, None]
    start = np.zeros((len(n), m, 3), dtype=np.float32)
    for b in range(len(n)):
        start[b, :n[b]] = _fcc(n[b], L[b])
    x = torch.tensor(start, device=dev)
    x = x + 0.04 * (2.0 * torch.rand(x.shape, device=dev, generator=gen) - 1.0)
    v = torch.randn(x.shape, device=dev, generator=gen) * real[:, :, None]
    v = (v - v.sum(1, keepdim=True) / nt[:, None, None]) * torch.sqrt(Tt)[:, None, None] * real[:, :, None]
    rc2 = rc * rc
    pair = real[:, :, None] & real[:, None, :] & ~torch.eye(m, dtype=torch.bool, device=dev)[None]
    far = torch.where(pair, 0.0, 2.0 * rc2)

    def force(x):
        d = [x[:, :, None, k] - x[:, None, :, k] for k in range(3)]
        d = [t - Lt[..., k] * torch.round(t / Lt[..., k]) for k, t in enumerate(d)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + far
        ir2 = 1.0 / r2.clamp_min(0.6)
        ir6 = ir2 * ir2 * ir2
        fr = 48.0 * ir6 * (ir6 - 0.5) * ir2 * (r2 < rc2)
        return torch.stack([(fr * t).sum(2) for t in d], 2)

    f = force(x)
    for s in range(MELT):
        v = v + 0.5 * DT * f
        x = x + DT * v
        f = force(x)
        v = v + 0.5 * DT * f
        if s % 20 == 19:
            v = v * torch.sqrt(3.0 * nt * Tt / (v * v).sum((1, 2)))[:, None, None]
    return [x[b, :n[b]].double() for b in range(len(n))]


def _repeat(tile, R, L):
    """R^3 copies of a tile that fill the box L (wrapped)."""
    dev = tile.device
    Lv = torch.tensor(L, device=dev)
    g = torch.stack(torch.meshgrid(*[torch.arange(R, device=dev, dtype=torch.float64)] * 3, indexing="ij"), -1)
    pos = (tile[None] + (g.reshape(-1, 1, 3) + 0.5) * (Lv / R) - 0.5 * Lv).reshape(-1, 3)
    return pos - Lv * torch.floor(pos / Lv + 0.5)


def _maxwell(n, T, gen):
    vel = torch.randn((n, 3), device=_dev(), dtype=torch.float64, generator=gen)
    vel -= vel.mean(0)
    vel *= math.sqrt(T * 3.0 * n) / vel.norm()
    return vel


def _box(n, rho, ay=1.0, az=1.0):
    a = np.array([1.0, ay, az])
    return a * (n / rho / float(np.prod(a))) ** (1.0 / 3.0)


def _state(n, rho, T, rc, seed, ay=1.0, az=1.0):
    """(pos, vel, L): a fluid of n atoms, device FP64 tensors."""
    dev = _dev()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + n)
    L = _box(n, rho, ay, az)
    R = 1
    while -(-n // R ** 3) > TILE:
        R += 1
    nt = -(-n // R ** 3)
    pos = _repeat(_melt([nt], [L / R], [T], rc, gen)[0], R, L)
    if pos.shape[0] > n:  # leave out a few, anywhere in the box
        pos = pos[torch.randperm(pos.shape[0], device=dev, generator=gen)[:n].sort().values]
    vel = _maxwell(n, T, gen)
    return pos.contiguous(), vel.contiguous(), L


def _replica_specs(case, seed):
    """(n, rho, T) of each replica: n log-uniform (the same for every seed,
    so that seeds cost alike), rho and T uniform, as in the ensemble
    configuration."""
    u = np.random.RandomState(int(seed) % (2 ** 31)).uniform(size=(case["replicas"], 2))
    return [(n, 0.6 + 0.4 * u[k, 0], 0.5 + 1.5 * u[k, 1]) for k, n in enumerate(_replica_sizes(case))]


def _replica_sizes(case):
    q = (np.arange(case["replicas"]) + 0.5) / case["replicas"]
    return np.exp(math.log(case["n_min"]) + math.log(case["n_max"] / case["n_min"]) * q).astype(int).tolist()


def _replica_states(case, seed):
    """The replicas' states on the host; their tiles (at most 512 atoms each)
    are melted side by side."""
    dev = _dev()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 17)
    specs = _replica_specs(case, seed)
    R = []
    for n, _, _ in specs:
        r = 1
        while -(-n // r ** 3) > 512:
            r += 1
        R.append(r)
    tiles = _melt([-(-n // r ** 3) for (n, _, _), r in zip(specs, R)],
                  [_box(n, rho) / r for (n, rho, _), r in zip(specs, R)], [T for _, _, T in specs], RC, gen)
    out = []
    for (n, rho, T), r, tile in zip(specs, R, tiles):
        L = _box(n, rho)
        pos = _repeat(tile, r, L)
        pos = pos[torch.randperm(pos.shape[0], device=dev, generator=gen)[:n].sort().values]
        vel = _maxwell(n, T, gen)
        out.append((pos.cpu().numpy().copy(), vel.cpu().numpy().copy(), L))
    return out


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------

ENERGIES = ("ke", "pe", "virial")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ensemble", "batch"):
        reps = _replica_states(case, seed)
        need = sum(md.md_ensemble_replica_bytes(md.replica_desc(L, len(p))) for p, _, L in reps)
        ens = md.Ensemble(need + (1 << 20), max_replicas=len(reps))
        # the shape that the autotuner takes for such replicas
        ens.set_shape(1024, 0, 2 if kind == "ensemble" else 8, 8192)
        st = dict(kind=kind, ens=ens, reps=reps, steps=case["steps"])
        if kind == "ensemble":
            st["ids"] = [ens.add(p, v, L) for p, v, L in reps]
            st["last"] = [p for p, _, _ in reps]
        return st
    if kind == "noalloc":
        pos, _, L = _state(case["n"], case["rho"], 1.0, case["rc"], seed)
        return dict(kind=kind, pos=pos, f=torch.zeros_like(pos), sums=torch.zeros(2, dtype=torch.float64, device=_dev()),
                    L=L, rc=case["rc"], n=case["n"])
    pos, vel, L = _state(case["n"], case["rho"], case["T"], case["rc"], seed, case.get("ay", 1.0), case.get("az", 1.0))
    ts = torch.cuda.Stream()
    ts.wait_stream(torch.cuda.current_stream())
    sim = md.Simulation(L, case["n"], case["rc"], case["skin"], DT, precision=case["form"],
                        cell_list_only=case.get("cells", False), stream=ts.cuda_stream)
    st = dict(kind=kind, sim=sim, ts=ts, pos=pos, vel=vel, L=torch.tensor(L, device=_dev()))
    if kind == "step":
        torch.cuda.current_stream().synchronize()
        sim.set_state(pos, vel)
        st.update(steps=case["steps"], last=pos, pos=torch.empty_like(pos), vel=torch.empty_like(vel))
        # positions as the library reports them (wrapped)
        sim.get_state(st["last"], st["vel"])
    return st


def run(state):
    kind = state["kind"]
    if kind == "step":
        sim, last, pos = state["sim"], state["last"], state["pos"]
        sim.step(state["steps"])
        m = sim.measure()
        with torch.cuda.stream(state["ts"]):
            sim.get_state(pos, state["vel"])
            moved = pos - last
            moved -= state["L"] * torch.round(moved / state["L"])
        state["last"], state["pos"] = pos, last
        return dict(moved=moved, vel=state["vel"], **{k: m[k] for k in ENERGIES})
    if kind == "load":
        sim = state["sim"]
        sim.set_state(state["pos"], state["vel"])
        m = sim.measure()
        return dict(f=sim.forces(), **{k: m[k] for k in ENERGIES})
    if kind == "noalloc":
        md.md_forces_noalloc(state["L"], state["n"], state["rc"], state["pos"].data_ptr(), state["f"].data_ptr(),
                             state["sums"].data_ptr(), stream=torch.cuda.current_stream().cuda_stream or None)
        return dict(f=state["f"], sums=state["sums"])
    ens, reps = state["ens"], state["reps"]
    ids = state["ids"] if kind == "ensemble" else [ens.add(p, v, L) for p, v, L in reps]
    ens.run(ids, state["steps"])
    moved, vels, sums = [], [], np.empty((len(ids), len(ENERGIES)))
    for k, (rid, (p0, _, L)) in enumerate(zip(ids, reps)):
        m = ens.measure(rid)
        sums[k] = [m[name] for name in ENERGIES]
        p, v = ens.get_state(rid)
        if kind == "ensemble":
            p0, state["last"][k] = state["last"][k], p
        else:
            ens.remove(rid)
        d = p - p0
        d -= L * np.rint(d / L)
        moved.append(d)
        vels.append(v)
    return dict(moved=np.concatenate(moved), vel=np.concatenate(vels), sums=sums)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how far results may be apart
# ---------------------------------------------------------------------------

def _pairs_per_atom(rho, rc):
    """Interacting pairs per atom (each counted once), from the density."""
    return 0.5 * rho * 4.0 / 3.0 * math.pi * rc ** 3


def work(case):
    """Bytes: the state (three FP64 position components, three velocities in
    the form's precision) read and written at every step; flops: 30 per
    interacting pair and 20 per atom for each step."""
    kind = case["kind"]
    if kind in ("ensemble", "batch"):
        atoms = float(sum(_replica_sizes(case)))
        return dict(bytes=atoms * (72.0 * case["steps"] + 96.0),
                    flops=atoms * case["steps"] * (30.0 * _pairs_per_atom(0.8, RC) + 20.0))
    pairs = 30.0 * _pairs_per_atom(case["rho"], case["rc"]) + 20.0
    n = float(case["n"])
    if kind == "step":
        state = 96.0 if case["form"] == "fp64" else 72.0
        return dict(bytes=n * (state * case["steps"] + 96.0), flops=n * case["steps"] * pairs)
    if kind == "load":
        return dict(bytes=n * (48.0 + 24.0), flops=n * pairs)
    return dict(bytes=n * 48.0, flops=n * pairs)


def tolerance(case):
    """About four times what the code shows against exact() at the start: a
    trajectory carries the rounding of its first steps into all that follow
    (FP32 pair terms: up to 3e-6 of the velocities after 100 steps; FP64: up
    to 4e-14 after 20, and ten times that is left for the order of sums)."""
    kind = case["kind"]
    if kind == "noalloc":
        return {"rel": 4e-13}
    if kind == "load":
        return {"rel": 4e-13 if case["form"] == "fp64" else 3e-6}
    if kind == "step" and case["form"] == "fp64":
        return {"rel": 4e-13}
    return {"rel": 1.2e-5, "max": 1e-3}


# ---------------------------------------------------------------------------
# the same results in 64 bits, with plain torch
# ---------------------------------------------------------------------------

def _find_pairs(x, sys, L, G, base, reach):
    """Pairs (i, j, image shift) with r < reach, each once; x wrapped,
    concatenated systems with boxes L[sys] and cell grids G[sys] whose cells
    start at base[sys]."""
    dev = x.device
    Ls, Gs = L[sys], G[sys]
    c = torch.minimum(((x / Ls + 0.5) * Gs).long(), Gs - 1).clamp_min(0)
    cid = base[sys] + (c[:, 2] * Gs[:, 1] + c[:, 1]) * Gs[:, 0] + c[:, 0]
    ncell = int((G.prod(1)).sum())
    order = torch.argsort(cid)
    count = torch.bincount(cid, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    occ = int(count.max())
    table = torch.full((ncell, occ), -1, dtype=torch.long, device=dev)
    table[cid[order], torch.arange(len(order), device=dev) - start[cid[order]]] = order
    csys = torch.repeat_interleave(torch.arange(len(G), device=dev), G.prod(1))
    cl = torch.arange(ncell, device=dev) - base[csys]
    cg = G[csys]
    cc = torch.stack([cl % cg[:, 0], (cl // cg[:, 0]) % cg[:, 1], cl // (cg[:, 0] * cg[:, 1])], 1)
    offs = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
            if (dz, dy, dx) >= (0, 0, 0)]
    got = []
    r2 = reach * reach
    step = max(1, (1 << 26) // (occ * occ))
    for off in offs:
        o = torch.tensor(off, device=dev)
        for b in range(0, ncell, step):
            s = slice(b, min(b + step, ncell))
            raw = cc[s] + o
            w = torch.div(raw, cg[s], rounding_mode="floor")
            nb = raw - w * cg[s]
            nid = base[csys[s]] + (nb[:, 2] * cg[s, 1] + nb[:, 1]) * cg[s, 0] + nb[:, 0]
            i = table[s][:, :, None].expand(-1, occ, occ)
            j = table[nid][:, None, :].expand(-1, occ, occ)
            ok = (i >= 0) & (j >= 0)
            if off == (0, 0, 0):
                ok &= i < j
            at = ok.nonzero()
            i, j = i[ok], j[ok]
            sh = -(w.double() * L[csys[s]])[at[:, 0]]
            d = x[i] - x[j] + sh
            near = (d * d).sum(1) < r2
            got.append((i[near], j[near], sh[near]))
    return tuple(torch.cat(t) for t in zip(*got))


def _pair_terms(x, i, j, sh, rc, shift):
    d = x[i] - x[j] + sh
    r2 = (d * d).sum(1)
    k = r2 < rc * rc
    d, r2, i, j = d[k], r2[k], i[k], j[k]
    ir2 = 1.0 / r2
    ir6 = ir2 ** 3
    fr = 48.0 * ir6 * (ir6 - 0.5) * ir2
    f = torch.zeros_like(x)
    g = fr[:, None] * d
    f.index_add_(0, i, g)
    f.index_add_(0, j, -g)
    return f, i, 4.0 * ir6 * (ir6 - 1.0) + shift, fr * r2


def _exact_run(systems, rc, steps):
    """Velocity Verlet in FP64 for concatenated systems [(pos, vel, L)]:
    displacements, velocities, forces and per-system (KE, PE, W) at the end."""
    dev = _dev()
    shift = 1.0 if abs(rc - RC) < 1e-9 else 0.0
    n = [p.shape[0] for p, _, _ in systems]
    x0 = torch.cat([torch.as_tensor(p, device=dev, dtype=torch.float64) for p, _, _ in systems])
    v = torch.cat([torch.as_tensor(w, device=dev, dtype=torch.float64) for _, w, _ in systems])
    L = torch.tensor(np.array([b for _, _, b in systems]), device=dev)
    sys = torch.repeat_interleave(torch.arange(len(n), device=dev), torch.tensor(n, device=dev))
    skin = min(0.6, float(L.min()) / 3.0 - rc)
    G = torch.clamp((L / (rc + skin)).floor().long(), min=3, max=400)
    cells = G.prod(1)
    base = torch.cumsum(cells, 0) - cells
    moved = torch.zeros_like(x0)
    anchor = None
    f = None
    for s in range(steps + 1):
        if s:
            v = v + 0.5 * DT * f
            moved = moved + DT * v
        if anchor is None or float(((moved - anchor) ** 2).sum(1).max()) > (0.5 * skin) ** 2:
            anchor = moved.clone()
            x = x0 + moved
            wrap = torch.floor(x / L[sys] + 0.5) * L[sys]
            i, j, sh = _find_pairs(x - wrap, sys, L, G, base, rc + skin)
        f, pi, u, w = _pair_terms(x0 + moved - wrap, i, j, sh, rc, shift)
        if s:
            v = v + 0.5 * DT * f
    sums = torch.zeros((len(n), 3), dtype=torch.float64, device=dev)
    sums[:, 0].index_add_(0, sys, 0.5 * (v * v).sum(1))
    sums[:, 1].index_add_(0, sys[pi], u)
    sums[:, 2].index_add_(0, sys[pi], w)
    return moved, v, f, sums


def exact(case, seed):
    kind = case["kind"]
    if kind in ("ensemble", "batch"):
        moved, v, _, sums = _exact_run(_replica_states(case, seed), RC, case["steps"])
        return dict(moved=moved.cpu().numpy(), vel=v.cpu().numpy(), sums=sums.cpu().numpy())
    pos, vel, L = _state(case["n"], case["rho"], case.get("T", 1.0), case["rc"], seed, case.get("ay", 1.0),
                         case.get("az", 1.0))
    if kind == "noalloc":
        _, _, f, sums = _exact_run([(pos, torch.zeros_like(pos), L)], case["rc"], 0)
        return dict(f=f, sums=sums[0, 1:])
    moved, v, f, sums = _exact_run([(pos, vel, L)], case["rc"], case.get("steps", 0))
    e = {k: float(sums[0, m]) for m, k in enumerate(ENERGIES)}
    if kind == "load":
        return dict(f=f.cpu().numpy(), **e)
    return dict(moved=moved, vel=v, **e)
