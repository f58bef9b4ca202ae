"""What a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public entry points (``paper_2504_21450_gb300.vlasov``,
``costmodel``, ``slab``) on inputs made from a seed on the GPU:

* ``advance``   load a state (per-cell block lists), run translation steps, read the state
                back: a run between two checkpoints, or one step of a coupled solver;
* ``dense``     the allocation-free step on caller-owned buffers;
* ``moments``   the velocity moments of every cell and the total mass (diagnostics);
* ``features``  the per-tile features and union counts the cost model reads;
* ``train``     full-batch training of the cost model;
* ``ghosts``    the coalesced ghost update of one z-slab (a rank's boundary planes read,
                its ghost planes replaced).

Distributions are drifting Maxwellians with cell-wise density noise: one population
everywhere ("uniform", every block above the threshold), or a beam and a hot sheath
joined by a front ("shock": across x; "front": rotated and rippled), which leaves most
of the velocity mesh empty.  The seed moves drifts, densities and fronts.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2504_21450_gb300 import costmodel, slab, vlasov

STORAGE = {"f32": vlasov.VL_STORE_F32, "bf16": vlasov.VL_STORE_BF16_SCALED,
           "f16": vlasov.VL_STORE_F16_SCALED}
FORM = {"fused": vlasov.VL_FORM_FUSED, "3pass": vlasov.VL_FORM_3PASS, "auto": vlasov.VL_FORM_AUTO}


def _grid(kind, name, n, nv, dv, dist, rel_thr, **more):
    c = {"kind": kind, "name": name, "nx": n[0], "ny": n[1], "nz": n[2],
         "nvx": nv[0], "nvy": nv[1], "nvz": nv[2], "dv": dv, "dist": dist, "rel_thr": rel_thr}
    c.update(more)
    return c


def _advance(name, n, nv, dv, dist, rel_thr, dt, steps, order="xyz", form="fused", storage="f32",
             graph=False):
    return _grid("advance", name, n, nv, dv, dist, rel_thr, dt=dt, steps=steps, order=order,
                 form=form, storage=storage, graph=graph)


def listed():
    return [
        # the smallest workload (8^3 cells, dense 16^3 velocity mesh), as a captured
        # sequence with the form left to the library: launches and latency count
        _advance("tiny_auto_graph", (8, 8, 8), (16, 16, 16), 1.0, "sine", 0.0, 0.1, 10, form="auto",
                 graph=True),
        # uniform-mesh scaling run (32^3 velocity mesh), default options: the largest
        _advance("uniform_fused", (64, 64, 16), (32, 32, 32), 1.0, "uniform", 1e-15, 0.05, 10),
        # the paper's sweep order z, x, y on extents that no tile divides
        _advance("ragged_zxy", (50, 37, 29), (24, 16, 16), 1.0, "uniform", 0.0, 0.05, 10, order="zxy"),
        # uneven sparsity: shock along x on a 64^3 velocity mesh, captured steps
        _advance("shock_graph", (128, 16, 16), (64, 64, 64), 1.0, "shock", 1e-5, 0.025, 8, graph=True),
        # classical per-direction form on a sparse state (rotated rippled front)
        _advance("front_3pass", (48, 48, 24), (64, 64, 64), 1.0, "front", 3e-4, 0.025, 8, form="3pass"),
        # classical form on a dense state
        _advance("uniform_3pass", (32, 32, 32), (32, 32, 32), 1.0, "uniform", 1e-15, 0.05, 10,
                 form="3pass"),
        # 16-bit storage on the precision workload's grid
        _advance("precision_bf16", (32, 32, 8), (32, 32, 32), 1.0, "uniform", 1e-15, 0.05, 10,
                 storage="bf16"),
        # one allocation-free step for a caller that owns all device memory
        _grid("dense", "dense_noalloc", (40, 32, 32), (16, 16, 16), 1.0, "uniform", 0.0, dt=0.1,
              order="xyz"),
        # diagnostics of a dense state: moments of every cell, total mass
        _grid("moments", "moments_mass", (64, 32, 16), (32, 32, 32), 1.0, "uniform", 1e-15,
              storage="f32"),
        # cost-model features of a sparse state, 8^3-cell tiles
        _grid("features", "tile_features", (48, 48, 24), (64, 64, 64), 1.0, "front", 3e-4, edge=8),
        # cost-model training on the number of samples two short traces give
        {"kind": "train", "name": "mlp_train", "samples": 5696, "epochs": 20},
        # ghost update of one z-slab: 3 boundary planes read and 3 ghost planes set, twice
        _grid("ghosts", "ghost_update", (32, 32, 22), (32, 32, 32), 1.0, "uniform", 1e-15),
    ]


def draw(rng):
    case = _drawn(rng)
    case.pop("name", None)
    return case


def _drawn(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def extents(cells, lo=6, hi=128):
        while True:
            n = [log_int(lo, hi) for _ in range(3)]
            if n[0] * n[1] * n[2] <= cells:
                return tuple(n)

    kind = rng.choice(["advance"] * 6 + ["dense", "moments", "features", "train", "ghosts"])
    if kind == "train":
        return {"kind": "train", "samples": log_int(500, 20000), "epochs": log_int(2, 20)}
    sparse = kind == "features" or (kind in ("advance", "moments") and rng.random() < 0.4)
    if sparse:
        dist = rng.choice(["shock", "front"])
        nv = rng.choice([(64, 64, 64), (48, 48, 48), (32, 32, 32)])
        rel = rng.choice([1e-5, 3e-4])
        dv = 64.0 / nv[0]
        n = extents(32768 if nv[0] > 32 else 65536, 8)
    else:
        dist, rel, dv = "uniform", 0.0, 1.0
        # (an allocation-free step's work list has room for about 1 MiB)
        nv = tuple(rng.choice([8, 16] if kind == "dense" else [8, 16, 24, 32]) for _ in range(3))
        n = extents(min(131072, 1_000_000_000 // (nv[0] * nv[1] * nv[2])))
    if kind == "ghosts":
        n = (n[0], n[1], max(n[2], 9))
        return _grid("ghosts", "", n, nv, dv, dist, rel)
    order = rng.choice(["xyz", "zxy", "yxz"])
    dt = rng.choice([0.25, 0.5, 0.8]) * 2.0 / (max(nv) * dv)
    if kind == "dense":
        return _grid("dense", "", n, nv, dv, dist, 0.0, dt=dt, order=order)
    storage = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
    if kind == "moments":
        return _grid("moments", "", n, nv, dv, dist, rel, storage=storage)
    if kind == "features":
        return _grid("features", "", n, nv, dv, dist, rel, edge=rng.choice([4, 8]))
    form = rng.choice(["fused", "fused", "3pass"])
    return _advance("", n, nv, dv, dist, rel, dt, rng.choice([1, 2, 4, 8]), order, form, storage,
                    rng.random() < 0.4)


# ---- inputs ------------------------------------------------------------------------------
def _n(case):
    return case["nx"], case["ny"], case["nz"]


def _nv(case):
    return case["nvx"], case["nvy"], case["nvz"]


def _vmin(case):
    return tuple(-0.5 * v * case["dv"] for v in _nv(case))


def _populations(case, r):
    """(density, drift, thermal speed) per population, drifts moved by up to a quarter."""
    def near(V):
        return tuple(float(v + 0.25 * case["dv"] * r.uniform(-1, 1)) for v in V)
    if case["dist"] in ("shock", "front"):
        return [(1.0, near((-8.0, 0.0, 0.0)), 1.5), (0.1, near((8.0, 0.0, 0.0)), 1.5),
                (4.0, near((-2.0, 0.0, 0.0)), 6.0)]
    s = 32.0 / max(_nv(case))  # drift and spread follow the width of the velocity mesh
    if case["dist"] == "sine":
        return [(1.0, near((0.5, 0.0, 0.0)), 2.0)]
    return [(1.0, near((2.0 / s, 1.0 / s, 0.0)), 3.0 / s)]


def _weights(case, r, dev):
    """Density of every population in every cell, [cells, populations] in 64 bits."""
    nx, ny, nz = _n(case)
    z, y, x = torch.meshgrid(*(torch.arange(m, dtype=torch.float64, device=dev) + 0.5
                               for m in (nz, ny, nx)), indexing="ij")
    gen = torch.Generator(device=dev).manual_seed(int(r.randint(1 << 30)))
    noise = 1.0 + 0.05 * (2.0 * torch.rand(nz * ny * nx, generator=gen, device=dev,
                                           dtype=torch.float64) - 1.0)
    shift = float(r.uniform(-2, 2))
    x, y = x.reshape(-1), y.reshape(-1)
    if case["dist"] == "sine":
        return (noise * (1.0 + 0.1 * torch.sin(2 * math.pi * (x + shift) / nx)))[:, None]
    if case["dist"] == "uniform":
        return noise[:, None]
    if case["dist"] == "shock":
        s = nx / (8.0 * math.pi) * torch.sin(2 * math.pi * (x - nx / 2 + shift) / nx)
    else:
        a = math.radians(30.0)
        xi = (x - nx / 2 + shift) * math.cos(a) + (y - ny / 2) * math.sin(a)
        eta = -(x - nx / 2 + shift) * math.sin(a) + (y - ny / 2) * math.cos(a)
        s = (xi - 3.0 * torch.sin(2 * math.pi * eta / 24.0 + float(r.uniform(0, 6.28)))) / 4.0
    up = 0.5 * (1.0 + torch.tanh(s))
    return torch.stack([noise * up, noise * 0.1 * up, noise * 4.0 * (1.0 - up)], dim=1)


def _shapes(case, pops, dev):
    """Value of every unit-density population in every velocity cell, [populations, ids, 64]."""
    nv, vmin, dv = _nv(case), _vmin(case), case["dv"]
    out = []
    for _, V, vth in pops:
        g = [torch.exp(-(vmin[d] + (torch.arange(nv[d], dtype=torch.float64, device=dev) + 0.5) * dv
                         - V[d]) ** 2 / (2 * vth * vth)) / (math.sqrt(2 * math.pi) * vth)
             for d in range(3)]
        G = g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
        G = G.reshape(nv[2] // 4, 4, nv[1] // 4, 4, nv[0] // 4, 4).permute(0, 2, 4, 1, 3, 5)
        out.append(G.reshape(-1, 64))
    return torch.stack(out)


def _state(case, seed, count_only=False):
    """Per-cell lists (off int64, ids int16, vals float32 [blocks, 64]) and the threshold."""
    dev = "cuda"
    r = np.random.RandomState(seed % (1 << 31))
    pops = _populations(case, r)
    w = _weights(case, r, dev)
    G = _shapes(case, pops, dev)
    thr = case["rel_thr"] * max(p[0] * float(G[k].max()) for k, p in enumerate(pops))
    ncell = w.shape[0]
    step = max(1, (1 << 27) // (G.shape[1] * 64))
    counts, ids, vals = [], [], []
    for s in range(0, ncell, step):
        f = torch.einsum("ck,kbv->cbv", w[s:s + step], G).to(torch.float32)
        keep = f.amax(dim=2).to(torch.float64) >= thr
        counts.append(keep.sum(dim=1))
        if not count_only:
            ci, bi = torch.nonzero(keep, as_tuple=True)
            ids.append(bi.to(torch.int16))
            vals.append(f[ci, bi])
    off = torch.zeros(ncell + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(counts), 0, out=off[1:])
    if count_only:
        return int(off[-1])
    return off, torch.cat(ids), torch.cat(vals), thr


def _samples(case, seed):
    """Tile features and targets of the cost model, with the spreads that traces have."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))
    n = case["samples"]

    def u(lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    blocks = u(6.0, 14.0)
    x = torch.stack([blocks, blocks + u(0.0, 0.8), u(0.1, 1.8), u(-9.0, 1.0), u(-0.5, 0.5),
                     u(-0.5, 0.5), u(1.4, 6.5), u(0.0, 0.4)], dim=1)
    t = x[:, 1] + 0.2 * x[:, 7] * x[:, 6] + 0.02 * torch.abs(x[:, 3])
    # the start of the parameters: uniform, scaled by fan-in and fan-out, biases 0
    r = np.random.RandomState(seed % (1 << 31))

    def layer(o, i):
        lim = math.sqrt(6.0 / (i + o))
        return r.uniform(-lim, lim, o * i)
    p = np.concatenate([layer(64, 8), np.zeros(64), layer(64, 64), np.zeros(64), layer(1, 64),
                        np.zeros(1)]).astype(np.float32)
    return x.to(torch.float32).contiguous(), t.to(torch.float32).contiguous(), p


def _new_grid(case, thr):
    return vlasov.Grid(_n(case), _nv(case), _vmin(case), (case["dv"],) * 3, threshold=thr,
                       storage=STORAGE[case.get("storage", "f32")])


# ---- one pass ----------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, p = _samples(case, seed)
        return {"case": case, "x": x, "t": t, "p": p}
    if kind == "dense":
        # the storage order of the call: [block id][vz in block][cell][vx + 4 vy]
        off, ids, vals, _ = _state(case, seed)
        ncell = off.numel() - 1
        nb = vals.shape[0] // ncell
        f = vals.view(ncell, nb, 4, 16).permute(1, 2, 0, 3).contiguous()
        n, nv, vmin = _n(case), _nv(case), _vmin(case)
        space = vlasov.vl_space_desc((ctypes.c_int * 3)(*n), (ctypes.c_double * 3)(1.0, 1.0, 1.0),
                                     (ctypes.c_double * 3)(0.0, 0.0, 0.0))
        vmesh = vlasov.vl_vmesh_desc((ctypes.c_int * 3)(*nv), (ctypes.c_double * 3)(*vmin),
                                     (ctypes.c_double * 3)(*((case["dv"],) * 3)),
                                     (ctypes.c_int * 3)(4, 4, 4))
        vlasov.load()
        return {"case": case, "f": f, "out": torch.empty_like(f), "space": space, "vmesh": vmesh,
                "mass": torch.zeros(1, dtype=torch.float64, device="cuda")}
    off, ids, vals, thr = _state(case, seed)
    g = _new_grid(case, thr)
    s = {"case": case, "grid": g}
    if kind == "advance":
        cap = _room(case)
        s.update(lists=(off, ids, vals), off=torch.empty_like(off), cap=cap,
                 ids=torch.zeros(cap, dtype=torch.int16, device="cuda"),
                 vals=torch.zeros((cap, 64), dtype=torch.float32, device="cuda"))
        return s
    g.set_blocks(off, ids, vals)
    if kind == "ghosts":
        s["slab"] = slab.Slab(0, 1, case["nz"] - 2 * slab.GHOST, 0, case["nz"] - 2 * slab.GHOST)
        s["planes"] = slab.GridPlanes(g)
    return s


def _room(case):
    """Blocks that the caller's buffers hold: those of the start and what the steps add."""
    m, full = _present(case), case["nx"] * case["ny"] * case["nz"] * _nb(case)
    return full if m == full else min(full, int(1.6 * m) + 1024)


def _nb(case):
    nv = _nv(case)
    return nv[0] * nv[1] * nv[2] // 64


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "advance":
        g = s["grid"]
        g.set_blocks(*s["lists"])
        g.translate(case["dt"], case["order"], case["steps"], form=FORM[case["form"]],
                    graph=case["graph"])
        vlasov.vl_get_blocks(g.handle, s["cap"], s["off"].data_ptr(), s["ids"].data_ptr(),
                             s["vals"].data_ptr(), 1)
        st = g.stats()
        # off[-1] blocks of the buffers are in use, the rest stay as the caller made them
        return {"off": s["off"], "ids": s["ids"], "vals": s["vals"], "mass": st.mass,
                "dropped_mass": st.dropped_mass}
    if kind == "dense":
        st = vlasov.vl_translate_dense_noalloc(
            s["space"], s["vmesh"], case["dt"], case["order"], 1, s["f"].data_ptr(),
            s["out"].data_ptr(), s["mass"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if st != vlasov.VL_OK:
            raise RuntimeError("vl_translate_dense_noalloc: " + vlasov.status_str(st))
        return {"f": s["out"], "mass": s["mass"]}
    if kind == "moments":
        g = s["grid"]
        return {"moments": g.moments(), "mass": g.mass()}
    if kind == "features":
        f, u = s["grid"].tile_features(case["edge"])
        return {"features": f, "union": u}
    if kind == "train":
        m = costmodel.CostModel(params=s["p"])
        losses = m.train(s["x"], s["t"], case["epochs"])
        return {"params": m.params, "m": m.m, "v": m.v, "losses": np.array(losses),
                "predicted": m.predict(s["x"])}
    p, sl = s["planes"], s["slab"]
    slab.ghost_update(sl, p.get, p.set, slab.loopback)
    lo, hi = p.get(0, slab.GHOST), p.get(sl.owned + slab.GHOST, slab.GHOST)
    return {"lo": lo, "hi": hi}


# ---- what a pass cannot do without -------------------------------------------------------
_blocks = {}


def _present(case):
    key = tuple(sorted((k, v) for k, v in case.items()
                       if k not in ("name", "kind", "steps", "order", "form", "graph", "storage", "dt", "edge")))
    if key not in _blocks:
        if case["dist"] in ("uniform", "sine"):
            _blocks[key] = case["nx"] * case["ny"] * case["nz"] * _nb(case)
        else:
            _blocks[key] = _state(case, 0, count_only=True)
    return _blocks[key]


def work(case):
    """Bytes: every input read once and every output written once, and the state read and
    written once per step (it does not fit on the chip).  Operations: 19 per value and
    sweep of a step (one push of the piecewise parabolic remap)."""
    kind = case["kind"]
    if kind == "train":
        per = 8 * 64 + 64 * 64 + 64
        return {"bytes": case["samples"] * 36.0 * case["epochs"] + 4801 * 24.0 * case["epochs"],
                "flops": 6.0 * case["samples"] * per * case["epochs"]}
    m = _present(case)
    v = m * 64.0
    stored = 4.0 if case.get("storage", "f32") == "f32" else 2.25
    if kind == "advance":
        return {"bytes": (4.0 + stored) * v * 2 + 2 * stored * v * case["steps"],
                "flops": 57.0 * v * case["steps"]}
    if kind == "dense":
        return {"bytes": 8.0 * v, "flops": 57.0 * v}
    if kind == "moments":
        return {"bytes": 2 * stored * v, "flops": 10.0 * v}
    if kind == "features":
        return {"bytes": 4.0 * v, "flops": 7.0 * v}
    plane = v / case["nz"]
    return {"bytes": 8.0 * plane * slab.GHOST * 6, "flops": 0.0}


# ---- the same in 64 bits, without the library --------------------------------------------
def _remap(a, dim, c):
    """One sweep: piecewise parabolic, semi-Lagrangian, |c| <= 1 cells, periodic along dim
    (Colella & Woodward 1984, face values kept between their two cells)."""
    up = c >= 0
    g = c.abs()
    nxt = torch.roll(a, -1, dim)
    face = (7.0 / 12.0) * (a + nxt) - (1.0 / 12.0) * (torch.roll(a, 1, dim) + torch.roll(a, -2, dim))
    face = torch.minimum(torch.maximum(face, torch.minimum(a, nxt)), torch.maximum(a, nxt))
    del nxt
    low = torch.roll(face, 1, dim)
    d1, d0 = torch.where(up, face - a, a - low), torch.where(up, a - low, face - a)
    del face, low
    # the edge the content leaves through is d1 away, the other one d0 (limiter 1.10)
    same = d1 * d0 > 0
    m1 = torch.where(d1.abs() > 2 * d0.abs(), 2 * d0, d1)
    m0 = torch.where(d0.abs() > 2 * d1.abs(), 2 * d1, d0)
    sgn = torch.where(up, 1.0, -1.0).to(a.dtype)
    zero = torch.zeros((), dtype=a.dtype, device=a.device)
    m1, m0 = torch.where(same, m1, zero), torch.where(same, m0, zero)
    out = g * (a + sgn * ((1 - g) * ((1 - g) * m1 + g * m0)))
    del d1, d0, m1, m0, same
    return a - out + torch.where(up, torch.roll(out, 1, dim), torch.roll(out, -1, dim))


def _advance64(case, off, ids, vals, thr, steps, order, dt):
    """The state after `steps` steps as (off, ids, vals): every block id by itself."""
    nx, ny, nz = _n(case)
    ncell, nv, vmin, dv, nb = nx * ny * nz, _nv(case), _vmin(case), case["dv"], _nb(case)
    dev = vals.device
    cell = torch.repeat_interleave(torch.arange(ncell, device=dev), off[1:] - off[:-1])
    idl = ids.to(torch.int64) & 0xffff
    by_id = torch.argsort(idl, stable=True)
    starts = torch.searchsorted(idl[by_id], torch.arange(nb + 1, device=dev)).tolist()
    group = max(1, (1 << 27) // (ncell * 64))
    active = [b for b in range(nb) if starts[b + 1] > starts[b]]
    thr32 = float(np.float32(thr))
    keys, parts = [], []
    for s in range(0, len(active), group):
        bs = active[s:s + group]
        F = torch.zeros((len(bs), ncell, 64), dtype=torch.float64, device=dev)
        P = torch.zeros((len(bs), ncell), dtype=torch.bool, device=dev)
        for j, b in enumerate(bs):
            at = by_id[starts[b]:starts[b + 1]]
            F[j, cell[at]] = vals[at].to(torch.float64)
            P[j, cell[at]] = True
        F = F.permute(0, 2, 1).reshape(len(bs), 4, 4, 4, nz, ny, nx).contiguous()
        P = P.view(len(bs), nz, ny, nx)
        bt = torch.tensor(bs, device=dev)
        bc = (bt % (nv[0] // 4), (bt // (nv[0] // 4)) % (nv[1] // 4), bt // (nv[0] // 4 * (nv[1] // 4)))
        cs = []
        for d in range(3):
            v = vmin[d] + ((4 * bc[d])[:, None] + torch.arange(4, device=dev) + 0.5).to(torch.float64) * dv
            sh = [len(bs), 1, 1, 1, 1, 1, 1]
            sh[3 - d] = 4
            cs.append((v * dt).view(sh))
        for _ in range(steps):
            for d in (1, 2, 3):
                P = P | torch.roll(P, 1, d) | torch.roll(P, -1, d)
            for ch in order:
                d = "xyz".index(ch)
                F = _remap(F, 6 - d, cs[d])
            keep = P & (F.amax(dim=(1, 2, 3)) >= thr32)
            F = F * keep[:, None, None, None]
            P = keep
        j, c = torch.nonzero(P.reshape(len(bs), ncell), as_tuple=True)
        keys.append(c * nb + bt[j])
        parts.append(F.reshape(len(bs), 64, ncell)[j, :, c])
        del F, P
    key = torch.cat(keys)
    key, at = torch.sort(key)
    return key, torch.cat(parts)[at]


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train64(case, seed)
    if kind == "ghosts":
        return None  # values are moved, not computed
    off, ids, vals, thr = _state(case, seed)
    ncell = off.numel() - 1
    if kind in ("advance", "dense"):
        steps = case.get("steps", 1)
        if ncell * 64.0 * _nb(case) * steps > 1.3e11:
            return None
        if case.get("storage", "f32") != "f32" and case["dist"] != "uniform":
            return None  # rounding moves blocks across the threshold
        key, v = _advance64(case, off, ids, vals, thr if kind == "advance" else 0.0, steps,
                            case["order"], case["dt"])
        mass = float(v.sum()) * case["dv"] ** 3
        if kind == "dense":
            return {"f": v.view(ncell, -1, 4, 16).permute(1, 2, 0, 3).contiguous(),
                    "mass": torch.tensor([mass], dtype=torch.float64)}
        vals = torch.zeros((_room(case), 64), dtype=torch.float64, device=v.device)
        vals[:v.shape[0]] = v
        return {"off": None, "ids": None, "vals": vals, "mass": mass, "dropped_mass": None}
    if kind == "moments" and case["storage"] != "f32":
        return None  # the moments are those of the rounded values
    mom = _moments64(case, off, ids, vals)
    if kind == "moments":
        return {"moments": mom, "mass": float(mom[:, 0].sum())}
    return {"features": _features64(case, off, ids, mom), "union": None}


def _moments64(case, off, ids, vals):
    """n, n V_d and P_dd of every cell: [cells, 7]."""
    ncell, nv, vmin, dv = off.numel() - 1, _nv(case), _vmin(case), case["dv"]
    dev = vals.device
    cell = torch.repeat_interleave(torch.arange(ncell, device=dev), off[1:] - off[:-1])
    out = torch.zeros((ncell, 7), dtype=torch.float64, device=dev)
    l = torch.arange(64, device=dev)
    inner = torch.stack([l & 3, (l >> 2) & 3, l >> 4], dim=1)

    def pieces():
        step = 1 << 21
        for s in range(0, vals.shape[0], step):
            b = ids[s:s + step].to(torch.int64) & 0xffff
            bc = torch.stack([b % (nv[0] // 4), (b // (nv[0] // 4)) % (nv[1] // 4),
                              b // (nv[0] // 4 * (nv[1] // 4))], dim=1)
            v = [vmin[d] + ((4 * bc[:, d])[:, None] + inner[:, d] + 0.5).to(torch.float64) * dv
                 for d in range(3)]
            yield cell[s:s + step], vals[s:s + step].to(torch.float64), v

    for c, f, v in pieces():
        out[:, 0].index_add_(0, c, f.sum(dim=1))
        for d in range(3):
            out[:, 1 + d].index_add_(0, c, (f * v[d]).sum(dim=1))
    V = out[:, 1:4] / torch.where(out[:, :1] != 0, out[:, :1], 1.0)
    for c, f, v in pieces():
        for d in range(3):
            out[:, 4 + d].index_add_(0, c, (f * (v[d] - V[c, d][:, None]) ** 2).sum(dim=1))
    return out * dv ** 3


def _features64(case, off, ids, mom):
    """The eight features of every tile (edge^3 cells, x fastest)."""
    nx, ny, nz = _n(case)
    e = case["edge"]
    nb, dev, ncell = _nb(case), mom.device, nx * ny * nz
    cell = torch.repeat_interleave(torch.arange(ncell, device=dev), off[1:] - off[:-1])
    P = torch.zeros((ncell, nb), dtype=torch.bool, device=dev)
    P[cell, ids.to(torch.int64) & 0xffff] = True
    U = P.view(nz, ny, nx, nb)
    for d in range(3):
        U = U | torch.roll(U, 1, d) | torch.roll(U, -1, d)
    act, uni = P.sum(dim=1), U.sum(dim=3).view(-1)
    c = torch.arange(ncell, device=dev)
    tx, ty = -(-nx // e), -(-ny // e)
    tile = (c % nx) // e + tx * (((c // nx) % ny) // e + ty * (c // (nx * ny) // e))
    nt = int(tile.max()) + 1
    n = mom[:, 0]
    safe = torch.where(n > 0, n, 1.0)
    V = mom[:, 1:4] / safe[:, None] * (n > 0)[:, None]
    vth = torch.sqrt(mom[:, 4:7].sum(dim=1) / (3 * safe)) * (n > 0)
    g2 = torch.zeros_like(n)
    for d in range(3):
        m = n.view(nz, ny, nx)
        g2 += (0.5 * (torch.roll(m, -1, 2 - d) - torch.roll(m, 1, 2 - d))).reshape(-1) ** 2
    grad = torch.sqrt(g2) / safe * (n > 0)

    def total(v):
        return torch.zeros(nt, dtype=torch.float64, device=dev).index_add_(0, tile, v.to(torch.float64))
    cnt = total(torch.ones_like(n))
    top = torch.zeros(nt, dtype=torch.float64, device=dev).scatter_reduce_(0, tile, grad, "amax")
    return torch.stack([torch.log1p(total(act)), torch.log1p(total(uni)), torch.log1p(total(n) / cnt)]
                       + [total(V[:, d]) / cnt for d in range(3)] + [total(vth) / cnt, top], dim=1)


def _train64(case, seed):
    """The epochs of full-batch Adam in 64 bits (constants as the 32-bit interface has them)."""
    x, t, p = _samples(case, seed)
    x, t = x.double(), t.double()
    p = torch.from_numpy(p).cuda().double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    b1, b2, lr, eps = 0.9, 0.999, 3e-3, 1e-8
    losses = []

    def net(q):
        w1, o = q[:512].view(64, 8), 512
        h = torch.relu(x @ w1.T + q[o:o + 64])
        o += 64
        h2 = torch.relu(h @ q[o:o + 4096].view(64, 64).T + q[o + 4096:o + 4160])
        o += 4160
        return h2 @ q[o:o + 64] + q[o + 64]

    for k in range(1, case["epochs"] + 1):
        q = p.clone().requires_grad_(True)
        loss = ((net(q) - t) ** 2).mean()
        grad, = torch.autograd.grad(loss, q)
        losses.append(float(loss))
        m = b1 * m + (1 - b1) * grad
        v = b2 * v + (1 - b2) * grad * grad
        p = p - lr * (m / (1 - b1 ** k)) / (torch.sqrt(v / (1 - b2 ** k)) + eps)
    return {"params": p, "m": m, "v": v, "losses": np.array(losses), "predicted": net(p)}
