"""Timed cases of the halo-finding library: what a program calls, at the sizes it calls it with.

A case is one call (or one graph replay) through the Python binding on buffers the program keeps: whole
finds from a small snapshot to the 1024^3 box, the multi-scale loop, a batch of subvolumes, and each stage
called on its own.  Inputs are clumped boxes (synth.py) drawn from a seed; fields and label grids that a
stage takes are made with plain torch.  exact() gives the same results in 64 bits with plain torch.
"""
import math

import torch

import paper_2501_10622_gb300 as pkg
from paper_2501_10622_gb300 import synth
from paper_2501_10622_gb300._lib import FRAC_BITS
from paper_2501_10622_gb300.batch import Batch, BatchJob

DEV = "cuda"
SPACING = 0.78125  # Mpc/h per cell: the cell size of served and batched jobs
FRAC = 1 << FRAC_BITS
CAT_CAP = 1 << 18  # catalogue rows a served slot keeps
BATCH_CAP = 1 << 13  # of one subvolume
ASSIGN_CAP = 1 << 16


def listed():
    return [
        # one small snapshot: launches and latency count
        {"name": "find-64", "kind": "find", "ng": 64, "np": 262144, "box": 50.0, "scales": 1, "masses": False},
        # a served job: 8 particles per cell
        {"name": "find-144-dense", "kind": "find", "ng": 144, "np": 23887872, "box": 144 * SPACING, "scales": 1,
         "masses": False},
        # the largest snapshot: 512^3 particles, 1024^3 grid, three wavelet scales
        {"name": "find-1024", "kind": "find", "ng": 1024, "np": 134217728, "box": 500.0, "scales": 3,
         "masses": False},
        # the paper's loop on its own 50 Mpc/h box and grid sizes Int(400 k_w + 150), with the self-boundness check
        {"name": "multiscale-190-590", "kind": "multiscale", "np": 16777216, "box": 50.0, "kw_high": 1.1, "scales": 6},
        # many uneven subvolumes in one CUDA graph
        {"name": "batch-24", "kind": "batch", "jobs": 24, "jobs_seed": 4, "ng_hi": 192, "np_hi": 1000000},
        # the mass grid of particles with masses of their own, on a ragged grid
        {"name": "deposit-242-masses", "kind": "deposit", "ng": 242, "np": 8388609, "box": 50.0, "masses": True},
        # one wavelet transform of a mass grid: a power of two, and two of the paper's sizes (2 5 19 and 2 281)
        {"name": "transform-512", "kind": "transform", "ng": 512, "box": 250.0, "w": 2.0},
        {"name": "transform-190", "kind": "transform", "ng": 190, "box": 50.0, "w": 2.0},
        {"name": "transform-562", "kind": "transform", "ng": 562, "box": 50.0, "w": 18.0},
        # segments of a given field
        {"name": "segment-384", "kind": "segment", "ng": 384, "box": 300.0, "w": 2.0},
        # particles to given segments, halo sums and catalogue
        {"name": "assign-256", "kind": "assign", "ng": 256, "np": 16777216, "box": 200.0, "w": 2.0, "masses": False},
        # the direct-space transform on a stencil (gdw_resolution of the paper's Table 1)
        {"name": "stencil-256", "kind": "stencil", "ng": 256, "box": 200.0, "w": 2.0, "R": 7},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    return 2 * round(_log(rng, lo, hi) / 2)


def draw(rng):
    kind = rng.choice(["find", "find", "multiscale", "batch", "deposit", "transform", "transform", "segment",
                       "assign", "stencil"])
    masses = rng.random() < 0.3
    w = round(rng.uniform(1.5, 4.0), 2)
    if kind == "find":  # grids of the form 2^a 3^b, as served jobs have
        ng = synth.smooth_ng(_log(rng, 32, 512))
        return {"kind": kind, "ng": ng, "np": int(min(ng ** 3 * _log(rng, 0.125, 8), 1 << 26)) | 1,
                "box": ng * SPACING, "scales": rng.randint(1, 3), "masses": masses}
    if kind == "multiscale":
        return {"kind": kind, "np": int(_log(rng, 1e5, 8e6)), "box": 50.0,
                "kw_high": round(rng.uniform(0.3, 0.9), 2), "scales": rng.randint(2, 5)}
    if kind == "batch":
        return {"kind": kind, "jobs": rng.randint(8, 32), "jobs_seed": rng.randrange(1 << 20),
                "ng_hi": rng.choice([96, 128, 192]), "np_hi": int(_log(rng, 1e5, 2e6))}
    if kind in ("deposit", "assign"):
        ng = _even(rng, 32, 512)
        d = {"kind": kind, "ng": ng, "np": int(min(ng ** 3 * _log(rng, 0.125, 8), 1 << 25)) | 1,
             "box": ng * SPACING, "masses": masses}
        return d if kind == "deposit" else dict(d, w=w)
    if kind == "stencil":
        ng = _even(rng, 32, 384)
        return {"kind": kind, "ng": ng, "box": ng * SPACING, "w": w, "R": rng.randint(3, 14)}
    ng = _even(rng, 32, 768 if kind == "transform" else 640)
    return {"kind": kind, "ng": ng, "box": ng * SPACING, "w": w}


def _scales(case):
    return [2.0, 3.0, 4.0][:case["scales"]]


def _ms_scales(case):
    _, ws, ngs = pkg.paper_scales(case["box"], 0.1, case["kw_high"], case["scales"])
    return ws, ngs


def _batch_shapes(case):
    grids = tuple(g for g in (32, 64, 96, 128, 192) if g <= case["ng_hi"])
    return synth.batched_subvolumes(case["jobs"], case["jobs_seed"], grids=grids, np_range=(1e4, case["np_hi"]))


def _particles(case, seed):
    """Positions, masses (or None) and their unit."""
    pos = synth.clumped_box(case["np"], case["box"], None, seed, DEV)
    if not case["masses"]:
        return pos, None, 1.0
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    n = case["np"]
    # 50 to 200 mass quanta per particle, fewer where the total would pass the library's 2^33
    top = min(200.0, 2.0 ** 32 / n)
    return pos, (0.25 + 0.75 * torch.rand(n, generator=gen, device=DEV)) * (0.01 * top), 0.01


def _mass_grid(case, seed):
    """The int64 mass grid of a clumped box with about one particle per 8 cells."""
    ng = case["ng"]
    pos = synth.clumped_box(max(1000, ng ** 3 // 8), case["box"], None, seed, DEV)
    return _cic(pos, None, 1.0, case["box"], ng)


def _field(case, seed):
    """A float32 wavelet field of a clumped box."""
    return _convolve(_mass_grid(case, seed), case["box"], case["w"], 1.0).float()


def _columns(cat):
    """The numbers of a catalogue buffer [..., cap, 64 bytes], by type."""
    return {"seed_n_part_n_cells": cat.view(torch.int64)[..., 0:3], "mass_centre": cat.view(torch.float64)[..., 3:7],
            "peak_last": cat.view(torch.float32)[..., 14]}


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "find":
        st["pos"], st["mass"], st["unit"] = _particles(case, seed)
        ns = case["scales"]
        st["ctx"] = pkg.Context(0, max_ng=case["ng"], max_np=case["np"], max_scales=ns)
        st["ctx"].prepare(case["ng"], case["box"], _scales(case))
        st["params"] = [pkg.default_params(w) for w in _scales(case)]
        st["halo_id"] = torch.empty((ns, case["np"]), dtype=torch.int32, device=DEV)
        st["cat"] = torch.zeros((ns, CAT_CAP, 64), dtype=torch.uint8, device=DEV)
        st["n_halo"] = torch.zeros(ns, dtype=torch.int64, device=DEV)
        st["out"] = {"halo_id": st["halo_id"], "n_halo": st["n_halo"], **_columns(st["cat"])}
    elif kind == "multiscale":
        n = case["np"]
        st["pos"], st["vel"] = synth.clumped_box(n, case["box"], 200, seed, DEV, velocities=True)
        st["ws"], st["ngs"] = _ms_scales(case)
        st["unit"] = synth.particle_mass(n, case["box"])
        st["ctx"] = pkg.Context(0, max_ng=max(st["ngs"]), max_np=n, max_scales=2, unbind=True)
        for w, ng in zip(st["ws"], st["ngs"]):
            st["ctx"].prepare(ng, case["box"], [w])
        st["halo_id"] = torch.empty(n, dtype=torch.int32, device=DEV)
        st["cat"] = torch.zeros((CAT_CAP, 64), dtype=torch.uint8, device=DEV)
        st["n_halo"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        st["out"] = {"halo_id": st["halo_id"], "n_halo": st["n_halo"],
                     "scale": st["cat"].view(torch.int32)[..., 15], **_columns(st["cat"])}
    elif kind == "batch":
        jobs = [BatchJob(synth.clumped_box(s.n_particles, s.box, s.n_clumps, seed * 1000 + i, DEV), s.box, s.ng,
                         [pkg.default_params(2.0)]) for i, s in enumerate(_batch_shapes(case))]
        st["batch"] = Batch(jobs, cat_cap=BATCH_CAP)
        # the program's own buffers, one for all jobs, in place of one per job
        ids = torch.empty((1, sum(j.np for j in jobs)), dtype=torch.int32, device=DEV)
        cat = torch.zeros((len(jobs), 1, BATCH_CAP, 64), dtype=torch.uint8, device=DEV)
        n_halo = torch.zeros((len(jobs), 1), dtype=torch.int64, device=DEV)
        at = 0
        for i, j in enumerate(jobs):
            j.halo_id, j.cat, j.n_halo = ids[:, at:at + j.np], cat[i], n_halo[i]
            at += j.np
        st["batch"].capture()
        st["out"] = {"halo_id": ids, "n_halo": n_halo, **_columns(cat)}
    elif kind == "deposit":
        st["pos"], st["mass"], st["unit"] = _particles(case, seed)
        st["ctx"] = pkg.Context(0, max_ng=case["ng"], max_np=case["np"], max_scales=1)
        st["grid"] = torch.empty((case["ng"],) * 3, dtype=torch.int64, device=DEV)
        st["mtot"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    elif kind in ("transform", "stencil"):
        st["grid"] = _mass_grid(case, seed)
        st["ctx"] = pkg.Context(0, max_ng=case["ng"], max_np=1, max_scales=1)
        st["ctx"].prepare(case["ng"], case["box"], [case["w"]])
        st["cwt"] = torch.empty((case["ng"],) * 3, dtype=torch.float32, device=DEV)
    elif kind == "segment":
        st["cwt"] = _field(case, seed)
        st["ctx"] = pkg.Context(0, max_ng=case["ng"], max_np=1, max_scales=1)
        st["label"] = torch.empty((case["ng"],) * 3, dtype=torch.int32, device=DEV)
    elif kind == "assign":
        st["pos"], st["mass"], st["unit"] = _particles(case, seed)
        st["cwt"] = _convolve(_cic(st["pos"], st["mass"], st["unit"], case["box"], case["ng"]), case["box"], case["w"],
                              st["unit"]).float()
        st["label"] = _segments(st["cwt"]).int()
        st["ctx"] = pkg.Context(0, max_ng=case["ng"], max_np=case["np"], max_scales=1)
        st["rows"] = torch.arange(ASSIGN_CAP, device=DEV)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "find":
        st["ctx"].find(st["pos"], case["box"], case["ng"], st["params"], mass=st["mass"], mass_unit=st["unit"],
                       cat_cap=CAT_CAP, halo_id=st["halo_id"], cat=st["cat"], n_halo=st["n_halo"])
        return st["out"]
    if kind == "multiscale":
        st["ctx"].find_multiscale(st["pos"], case["box"], st["ws"], st["ngs"], mass_unit=st["unit"], vel=st["vel"],
                                  cat_cap=CAT_CAP, halo_id=st["halo_id"], cat=st["cat"], n_halo=st["n_halo"])
        return st["out"]
    if kind == "batch":
        st["batch"].replay()
        return st["out"]
    if kind == "deposit":
        return st["ctx"].deposit(st["pos"], case["box"], case["ng"], mass=st["mass"], mass_unit=st["unit"],
                                 grid=st["grid"], mtot=st["mtot"]), st["mtot"]
    if kind == "transform":
        return st["ctx"].transform(st["grid"], case["box"], case["w"], cwt=st["cwt"])
    if kind == "stencil":
        return st["ctx"].transform_stencil(st["grid"], case["box"], case["w"], case["R"], cwt=st["cwt"])
    if kind == "segment":
        return st["ctx"].segment(st["cwt"], label=st["label"])
    halo_id, cat, n_halo = st["ctx"].assign(st["pos"], case["box"], st["label"], cwt=st["cwt"], mass=st["mass"],
                                            mass_unit=st["unit"], cat_cap=ASSIGN_CAP)
    # the buffer is a fresh one: only the halos found are the caller's
    found = st["rows"] < n_halo
    return {"halo_id": halo_id, "n_halo": n_halo,
            **_columns(torch.where(found[:, None], cat.view(torch.int64), 0).view(torch.uint8))}


def _find_work(ng, n, scales, masses):
    """One find: positions (and masses) in, halo ids out; the arithmetic of the deposit (8 nodes per particle), a
    forward and per scale an inverse real FFT, 26 comparisons per cell and scale, the halo sums."""
    cells = ng ** 3
    fft = 2.5 * cells * math.log2(cells)
    return {"bytes": (16 if masses else 12) * n + 4 * n * scales,
            "flops": 40 * n + fft + scales * (fft + 30 * cells + 10 * n)}


def work(case):
    kind = case["kind"]
    if kind == "find":
        return _find_work(case["ng"], case["np"], case["scales"], case["masses"])
    if kind == "batch":
        ws = [_find_work(s.ng, s.n_particles, 1, False) for s in _batch_shapes(case)]
        return {k: sum(x[k] for x in ws) for k in ("bytes", "flops")}
    if kind == "multiscale":  # positions, velocities in, ids out; every scale has a grid and a deposit of its own
        n = case["np"]
        ws = [_find_work(g, n, 1, False)["flops"] for g in _ms_scales(case)[1]]
        return {"bytes": (12 + 12 + 4) * n, "flops": sum(ws)}
    cells = case["ng"] ** 3
    if kind == "deposit":
        return {"bytes": (16 if case["masses"] else 12) * case["np"] + 8 * cells, "flops": 40 * case["np"]}
    if kind == "transform":
        return {"bytes": 12 * cells, "flops": 5.0 * cells * math.log2(cells) + cells}
    if kind == "stencil":
        return {"bytes": 12 * cells, "flops": cells * 7 * 3 * case["R"]}
    if kind == "segment":
        return {"bytes": 8 * cells, "flops": 30 * cells}
    return {"bytes": (16 if case["masses"] else 12) * case["np"] + 4 * case["np"] + 4 * cells,
            "flops": 10 * case["np"]}


# ---- the same results in 64 bits, with plain torch ----------------------------

def _quantised(pos, box, ng):
    """Fixed-point coordinates: floor(x s) mod ng 2^10, s = ng / box 2^10 rounded to 29 bits (exact products)."""
    f, e = math.frexp(ng / box * FRAC)
    s = math.ldexp(round(math.ldexp(f, 29)), e - 29)
    return torch.floor(pos.double() * s).long() % (ng * FRAC)


def _quanta(mass, unit, n):
    return torch.ones(n, dtype=torch.int64, device=DEV) if mass is None else torch.round(mass.double() / unit).long()


def _cic(pos, mass, unit, box, ng):
    grid = torch.zeros(ng ** 3, dtype=torch.int64, device=DEV)
    for p in range(0, pos.shape[0], 1 << 24):
        q = _quantised(pos[p:p + (1 << 24)], box, ng)
        mq = _quanta(None if mass is None else mass[p:p + (1 << 24)], unit, q.shape[0])
        node, frac = q // FRAC, q % FRAC
        for c in range(8):
            wt, cell = mq, 0
            for d in (2, 1, 0):
                up = (c >> d) & 1
                wt = wt * (frac[:, d] if up else FRAC - frac[:, d])
                cell = cell * ng + (node[:, d] + up) % ng
            grid.index_add_(0, cell, wt)
    return grid.view(ng, ng, ng)


def _convolve(grid, box, w, unit, R=None):
    """The wavelet transform in fp64: the Mexican hat sampled at minimum-image offsets (within R cells if given)."""
    ng = grid.shape[0]
    d = torch.arange(ng, device=DEV, dtype=torch.float64)
    d = torch.where(2 * d <= ng, d, d - ng)
    u2 = (w * box / ng * d) ** 2
    g = torch.exp(-0.25 * u2)
    if R is not None:
        g = torch.where(d.abs() <= R, g, torch.zeros_like(g))
    G, H = torch.fft.fft(g).real, torch.fft.fft(u2 * g).real
    half = ng // 2 + 1
    gx, gy, gz = G[None, None, :half], G[None, :, None], G[:, None, None]
    hx, hy, hz = H[None, None, :half], H[None, :, None], H[:, None, None]
    spec = torch.fft.rfftn(grid.double() * (unit * 2.0 ** -30))
    spec *= w ** 1.5 * (gz * (6 * gx * gy - hx * gy - gx * hy) - hz * (gx * gy))
    return torch.fft.irfftn(spec, s=grid.shape)


def _segments(field):
    """Labels: every cell takes the seed (a maximum above 0) that steepest ascent over 26 neighbours reaches, or -1."""
    ng = field.shape[0]
    idx = torch.arange(ng ** 3, device=DEV).view(ng, ng, ng)
    best, arg = field.clone(), idx.clone()
    for k in range(27):
        sh = (k // 9 - 1, k // 3 % 3 - 1, k % 3 - 1)
        v, j = torch.roll(field, sh, (0, 1, 2)), torch.roll(idx, sh, (0, 1, 2))
        win = (v > best) | ((v == best) & (j < arg))
        best, arg = torch.where(win, v, best), torch.where(win, j, arg)
    p = arg.view(-1)
    while True:
        q = p[p]
        if torch.equal(p, q):
            break
        p = q
    return torch.where(field.view(-1)[p] > 0, p, torch.full_like(p, -1)).view(ng, ng, ng)


def _halos(pos, mass, unit, box, label, field, cap):
    """Halo ids and the catalogue's numbers, padded with zeros to cap rows."""
    ng = label.shape[0]
    lab = label.reshape(-1).long()
    q, mq = _quantised(pos, box, ng), _quanta(mass, unit, pos.shape[0])
    node = (q + FRAC // 2) // FRAC % ng
    plab = lab[(node[:, 2] * ng + node[:, 1]) * ng + node[:, 0]]
    seeds = torch.nonzero(lab == torch.arange(ng ** 3, device=DEV)).view(-1)
    slot_of = torch.full((ng ** 3 + 1,), -1, dtype=torch.int64, device=DEV)
    slot_of[seeds] = torch.arange(len(seeds), device=DEV)
    cells = torch.bincount(slot_of[lab[lab >= 0]], minlength=len(seeds))
    inh = plab >= 0
    slot, q, mq = slot_of[plab[inh]], q[inh], mq[inh]
    n_part = torch.bincount(slot, minlength=len(seeds))
    m = torch.zeros(len(seeds), dtype=torch.int64, device=DEV).index_add_(0, slot, mq)
    sc = torch.stack([seeds % ng, seeds // ng % ng, seeds // (ng * ng)], 1)
    M = ng * FRAC
    dq = (q - sc[slot] * FRAC + M // 2) % M - M // 2
    mom = torch.zeros((len(seeds), 3), dtype=torch.int64, device=DEV).index_add_(0, slot, mq[:, None] * dq)
    total = float(_quanta(mass, unit, pos.shape[0]).sum())
    keep = (n_part >= 15) & (m.double() * float(ng ** 3) >= (4.0 * total) * cells.double())
    k = torch.nonzero(keep).view(-1)
    centre = ((sc[k] * FRAC).double() + mom[k].double() / m[k].double()[:, None]) * (box / ng / FRAC)
    centre = torch.where(centre >= box, centre - box, torch.where(centre < 0, centre + box, centre))
    halo_id = torch.full_like(plab, -1)
    halo_id[inh] = torch.where(keep, seeds, torch.full_like(seeds, -1))[slot]
    out = {"seed_n_part_n_cells": torch.zeros((cap, 3), dtype=torch.int64, device=DEV),
           "mass_centre": torch.zeros((cap, 4), dtype=torch.float64, device=DEV),
           "peak_last": torch.zeros(cap, dtype=torch.float64, device=DEV)}
    n = len(k)
    out["seed_n_part_n_cells"][:n] = torch.stack([seeds[k], n_part[k], cells[k]], 1)
    out["mass_centre"][:n] = torch.cat([(m[k].double() * unit)[:, None], centre], 1)
    out["peak_last"][:n] = field.reshape(-1)[seeds[k]].double()
    return {"halo_id": halo_id, "n_halo": torch.tensor([n], device=DEV), **out}


def _exact_find(pos, mass, unit, box, ng, ws, cap):
    """The floating columns of a find (its whole numbers hang on near ties of the field's 32 bits: no value here)."""
    grid = _cic(pos, mass, unit, box, ng)
    res = []
    for w in ws:
        field = _convolve(grid, box, w, unit)
        res.append(_halos(pos, mass, unit, box, _segments(field), field, cap))
    return {"halo_id": None, "n_halo": None, "seed_n_part_n_cells": None,
            **{k: torch.stack([r[k] for r in res]) for k in ("mass_centre", "peak_last")}}


def exact(case, seed):
    kind = case["kind"]
    if kind == "find":
        if case["ng"] > 384:
            return None  # too large for torch's intermediates
        pos, mass, unit = _particles(case, seed)
        return _exact_find(pos, mass, unit, case["box"], case["ng"], _scales(case), CAT_CAP)
    if kind == "batch":
        res = [_exact_find(synth.clumped_box(s.n_particles, s.box, s.n_clumps, seed * 1000 + i, DEV), None, 1.0,
                           s.box, s.ng, [2.0], BATCH_CAP) for i, s in enumerate(_batch_shapes(case))]
        return {k: None if v is None else torch.stack([r[k] for r in res]) for k, v in res[0].items()}
    if kind == "deposit":
        pos, mass, unit = _particles(case, seed)
        return (_cic(pos, mass, unit, case["box"], case["ng"]), _quanta(mass, unit, case["np"]).sum().view(1))
    if kind == "transform":
        return _convolve(_mass_grid(case, seed), case["box"], case["w"], 1.0)
    if kind == "stencil":
        return _convolve(_mass_grid(case, seed), case["box"], case["w"], 1.0, case["R"])
    if kind == "segment":
        return _segments(_field(case, seed)).int()
    if kind == "assign":
        pos, mass, unit = _particles(case, seed)
        field = _convolve(_cic(pos, mass, unit, case["box"], case["ng"]), case["box"], case["w"], unit).float()
        return _halos(pos, mass, unit, case["box"], _segments(field), field, ASSIGN_CAP)
    return None  # multiscale: the loop with its self-boundness check takes minutes in plain torch
