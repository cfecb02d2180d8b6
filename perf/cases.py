"""Timed cases of the QED step: what a program that uses this package calls in
its main loop, over the range of sizes, precisions and options it is used with.

A case is a dict of plain values; prepare() makes what a program holds before
the call, run() is one pass through the public entry points.  A pass that
recoils or consumes particles first puts the momenta (and, on a grid, the
positions), the alive flags and the counts back from a device copy, as the
benchmark's fixed-work steps do, so that every pass does the same work.

Photons appended in any order (order "any") are the same set in an order that
depends on the scheduling of the GPU, so those cases return the leptons, the
pairs, the photons that were there and the counts; the cases with ordered
appends return the new photons too.
"""
from __future__ import annotations

import math
from collections import OrderedDict

import torch

from paper_1608_06356_gb300 import api

A_S = 412148.45          # Schwinger field in field units at 1 um
DT = 0.01
STATE = ("x", "y", "z", "px", "py", "pz")
FIELDS = ("ex", "ey", "ez", "bx", "by", "bz")
GRID_DX = 2 * math.pi / 32  # cascade grid: 32 cells per wavelength
PIC_DX, PIC_DT, PIC_DENSITY, PIC_P_TH = 0.25, 0.1, 0.05, 0.02


def listed():
    return [
        # the paper's single-particle-type test (gamma0 = 1000, B = 410, chi ~ 1) in FP64, push and
        # emission as separate calls: the smallest call, ten thousand electrons per launch
        {"name": "single_fp64_10k", "kind": "uniform", "n": 10_000, "precision": 64, "generator": 0, "order": "ordered"},
        # the uniform-field ensemble: a million electrons and as many photons with fields of their
        # own, emission and pairs; the ordinary step of a cascade study without a grid
        {"name": "ensemble_1m", "kind": "ensemble", "n": 1 << 20, "order": "any"},
        # the headline ensemble, 64M electrons over five decades of chi: the largest call
        {"name": "chi_64m_any", "kind": "chi", "n": 1 << 26, "order": "any", "sampler": "table"},
        # the same ensemble at 4M through the default, reproducible append order
        {"name": "chi_4m_ordered", "kind": "chi", "n": 1 << 22, "order": "ordered", "sampler": "table"},
        # the learned sampler in the step
        {"name": "chi_4m_mlp", "kind": "chi", "n": 1 << 22, "order": "any", "sampler": "mlp"},
        # a mid-cascade step in the 256^3 standing wave: the field of the step's time, CIC gather,
        # electrons, positrons and photons in the central block
        {"name": "cascade_256", "kind": "cascade", "nx": 256, "ny": 256, "nz": 256, "n": 1 << 21, "order": "any"},
        # one cycle of the self-consistent loop, particles stored by cell, eight per cell
        {"name": "pic_128_cells", "kind": "pic", "nx": 128, "ny": 128, "nz": 128, "ppc": 8, "cell_order": True},
        # the same on a grid larger than L2 with particles in random order (a program that does not sort)
        {"name": "pic_256_random", "kind": "pic", "nx": 256, "ny": 256, "nz": 256, "ppc": 1, "cell_order": False},
        # many uneven runs advanced together under a graph: a scan over chi
        {"name": "batched_64", "kind": "batched", "runs": 64, "lo": 1000, "hi": 200_000, "steps": 4},
        # leptons kept in host memory and streamed through the GPU
        {"name": "host_4m", "kind": "host", "n": 1 << 22, "chunk": 1 << 19},
        # removal of the photons that made pairs, between steps (keeps the order)
        {"name": "compact_8m", "kind": "compact", "n": 1 << 23, "dead": 0.1, "fields": True, "precision": 32},
        # training of the learned sampler: load, 16 optimiser steps, read the weights
        {"name": "train_16", "kind": "train", "samples": 16 * 38912},
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]; odd three times in four."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(v | 1, hi) if rng.random() < 0.75 else v


def draw(rng):
    kind = rng.choice(("uniform", "ensemble", "chi", "chi", "cascade", "pic", "pic", "batched", "host", "compact",
                       "train"))
    order = rng.choice(("any", "ordered"))
    if kind == "uniform":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 20), "precision": rng.choice((32, 64)),
                "generator": rng.choice((0, 0, 1, 2)), "order": "ordered"}
    if kind == "ensemble":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 22), "order": order}
    if kind == "chi":
        sampler = rng.choice(("table", "table", "mlp"))
        return {"kind": kind, "n": _log_int(rng, 10_000, 1 << 24), "order": order, "sampler": sampler}
    if kind == "cascade":
        nx, ny, nz = (rng.choice((64, 96, 129, 192, 250)) for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "n": _log_int(rng, 10_000, 1 << 21), "order": order}
    if kind == "pic":
        nx, ny, nz = (_log_int(rng, 24, 200) for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "ppc": rng.choice((1, 2, 4)),
                "cell_order": rng.random() < 0.6}
    if kind == "batched":
        return {"kind": kind, "runs": _log_int(rng, 8, 128), "lo": 1000, "hi": _log_int(rng, 20_000, 200_000),
                "steps": rng.choice((2, 4))}
    if kind == "host":
        n = _log_int(rng, 100_000, 1 << 22)
        return {"kind": kind, "n": n, "chunk": max(4096, n // rng.choice((4, 8, 16)))}
    if kind == "compact":
        return {"kind": kind, "n": _log_int(rng, 10_000, 1 << 24), "dead": rng.choice((0.01, 0.1, 0.5)),
                "fields": rng.random() < 0.5, "precision": rng.choice((32, 64))}
    return {"kind": "train", "samples": 38912 * rng.choice((4, 8, 16))}


# ---- contexts ---------------------------------------------------------------
# A program builds its tables once and keeps the context; the last few
# configurations are kept here for the same reason.
_contexts: OrderedDict = OrderedDict()


def _new_context(**cfg):
    ctx = api.qed_init_tables(api.config(**cfg))
    if cfg.get("sampler"):
        api.qed_mlp_load(ctx, api.mlp_init_params(0))
    return ctx


def _context(**cfg):
    key = tuple(sorted(cfg.items()))
    ctx = _contexts.pop(key, None)
    if ctx is None:
        ctx = _new_context(**cfg)
        while len(_contexts) >= 4:
            _contexts.popitem(last=False)
    _contexts[key] = ctx
    return ctx


# ---- inputs -----------------------------------------------------------------
class _Rand:
    def __init__(self, seed, device="cuda"):
        self.g = torch.Generator(device=device).manual_seed(int(seed))
        self.device = device

    def uniform(self, n, lo=0.0, hi=1.0, dtype=torch.float32):
        return torch.rand(n, generator=self.g, device=self.device, dtype=dtype) * (hi - lo) + lo

    def log_uniform(self, n, lo, hi, dtype=torch.float32):
        return torch.exp(self.uniform(n, math.log(lo), math.log(hi), dtype))

    def iso(self, n, dtype=torch.float32):
        mu, phi = self.uniform(n, -1.0, 1.0, dtype), self.uniform(n, 0.0, 2 * math.pi, dtype)
        s = torch.sqrt(1.0 - mu * mu)
        return torch.stack([s * torch.cos(phi), s * torch.sin(phi), mu])

    def normal(self, n, dtype=torch.float32):
        return torch.randn(n, generator=self.g, device=self.device, dtype=dtype)

    def id0(self):
        return int(torch.randint(0, 1 << 40, (1,), generator=self.g, device=self.device))


def _species(cap, q, dtype=torch.float32, fields=False, rows=STATE[3:], **kw):
    """A species whose `rows` arrays are rows of one buffer (each 512-byte
    aligned), so that one device copy restores them.  Returns (species, buffer)."""
    s = api.Species.empty(cap, q, dtype=dtype, fields=fields, **kw)
    buf = torch.zeros((len(rows), (cap + 127) // 128 * 128), dtype=dtype, device="cuda")
    for k, name in enumerate(rows):
        setattr(s, name, buf[k, :cap])
    return s, buf


def _counts(*species):
    """The species' counts as elements of one device tensor."""
    n = torch.zeros(len(species), dtype=torch.int64, device="cuda")
    for k, s in enumerate(species):
        s.n = n[k:k + 1]
    return n


def _fill(s, n, **arrays):
    for name, a in arrays.items():
        getattr(s, name)[:n].copy_(a)
    if s.alive is not None:
        s.alive[:n] = 1
    s.n.fill_(n)


def _ids(r, n):
    a = r.id0()
    return torch.arange(a, a + n, dtype=torch.int64, device="cuda")


def _vec(names, v):
    return dict(zip(names, v))


def _chi_particles(r, n, chi_lo, chi_hi, g_lo=1e2, g_hi=1e4):
    """gamma and chi log-uniform, isotropic directions, B perpendicular to p
    with |B| = chi a_S / |p|, E = 0."""
    g = r.log_uniform(n, g_lo, g_hi)
    chi = r.log_uniform(n, chi_lo, chi_hi) if isinstance(chi_lo, float) else \
        torch.exp(r.uniform(n) * torch.log(chi_hi / chi_lo) + torch.log(chi_lo))
    d, b = r.iso(n), r.iso(n)
    b -= d * (b * d).sum(0)
    b *= chi * A_S / torch.sqrt(g * g - 1.0) / torch.linalg.vector_norm(b, dim=0)
    return torch.sqrt(g * g - 1.0) * d, b


def _seed_of(case):
    return 1 + sum(map(ord, case["kind"]))


def _prepare_uniform(case, seed):
    n, f64 = case["n"], case["precision"] == 64
    dtype = torch.float64 if f64 else torch.float32
    cap_g = n + 4096
    ctx = _context(dt=DT, seed=_seed_of(case), precision=int(f64), generator=case["generator"],
                   append_order=0, max_particles=max(cap_g, 1 << 16))
    r = _Rand(seed)
    od = case["generator"] != 0
    e, buf = _species(n, -1, dtype, od=od)
    g = api.Species.empty(cap_g, 0, dtype=dtype)
    phi = r.uniform(n, 0.0, 2 * math.pi, torch.float64)
    p0 = math.sqrt(1000.0 ** 2 - 1.0)
    _fill(e, n, px=p0 * torch.cos(phi), py=p0 * torch.sin(phi), w=torch.ones(n, device="cuda"), id=_ids(r, n))
    return {"ctx": ctx, "e": e, "g": g, "buf": buf, "buf0": buf.clone(), "step": 0,
            "f": api.Fields.uniform((0.0, 0.0, 0.0), (0.0, 0.0, 410.0))}


def _run_uniform(s):
    s["buf"].copy_(s["buf0"])
    s["g"].n.zero_()
    api.qed_gather_push(s["ctx"], s["e"], s["f"], s["step"])
    api.qed_emit(s["ctx"], s["e"], s["g"], s["f"], s["step"])
    s["step"] += 1
    return {"e": _arrays(s["e"], STATE), "g": _arrays(s["g"], STATE + ("w", "id")), "n": s["g"].n}


def _arrays(sp, names):
    return {k: getattr(sp, k) for k in names if getattr(sp, k) is not None}


def _prepare_ensemble(case, seed):
    n = case["n"]
    cap, cap_g = n + n // 4 + 4096, 2 * n + 4096
    ctx = _context(dt=DT, seed=_seed_of(case), append_order=int(case["order"] == "any"), max_particles=max(cap_g, 1 << 16))
    r = _Rand(seed)
    e, buf = _species(cap, -1, fields=True)
    p = api.Species.empty(cap - n, 1, fields=True)
    g = api.Species.empty(cap_g, 0, fields=True)
    cnt = _counts(e, p, g)
    for s, photon in ((e, False), (g, True)):
        gam = r.log_uniform(n, 1e2, 1e4)
        mom = (gam if photon else torch.sqrt(gam * gam - 1.0)) * r.iso(n)
        _fill(s, n, **_vec(STATE[:3], (r.uniform(n, -1.0, 1.0) for _ in range(3))), **_vec(STATE[3:], mom),
              **_vec(FIELDS[:3], r.iso(n) * r.log_uniform(n, 10.0, 2000.0)),
              **_vec(FIELDS[3:], r.iso(n) * r.log_uniform(n, 10.0, 2000.0)),
              w=torch.ones(n, device="cuda"), id=_ids(r, n))
    return {"ctx": ctx, "e": e, "p": p, "g": g, "buf": buf, "buf0": buf.clone(), "alive0": g.alive[:n].clone(),
            "cnt": cnt, "cnt0": cnt.clone(), "n": n, "any": case["order"] == "any", "step": 0,
            "f": api.Fields.per_particle()}


def _restore(s):
    s["buf"].copy_(s["buf0"])
    s["cnt"].copy_(s["cnt0"])


def _run_ensemble(s):
    _restore(s)
    s["g"].alive[:s["n"]].copy_(s["alive0"])
    api.qed_step_fused(s["ctx"], s["e"], s["p"], s["g"], s["f"], s["step"])
    s["step"] += 1
    kept = STATE + ("w", "id") + FIELDS
    g = _arrays(s["g"], STATE[:3] + ("alive",) if s["any"] else kept + ("alive",))
    if s["any"]:  # the photons that were there; the new ones behind them have no order
        g = {k: v[:s["n"]] for k, v in g.items()}
    return {"e": _arrays(s["e"], kept), "p": _arrays(s["p"], kept), "g": g, "n": s["cnt"]}


def _prepare_chi(case, seed):
    n = case["n"]
    cap, cap_p, cap_g = n + n // 8 + 64, n // 8 + 64, int(0.3 * n) + 4096
    ctx = _context(dt=DT, seed=_seed_of(case), append_order=int(case["order"] == "any"),
                   sampler=int(case["sampler"] == "mlp"), max_particles=max(cap, 1 << 16))
    r = _Rand(seed)
    e, buf = _species(cap, -1, fields=True)
    p = api.Species.empty(cap_p, 1, fields=True)
    g = api.Species.empty(cap_g, 0, fields=True)
    cnt = _counts(e, p, g)
    mom, b = _chi_particles(r, n, 1e-3, 1e2)
    _fill(e, n, **_vec(STATE[3:], mom), **_vec(FIELDS[3:], b), w=torch.ones(n, device="cuda"), id=_ids(r, n))
    return {"ctx": ctx, "e": e, "p": p, "g": g, "buf": buf, "buf0": buf.clone(), "cnt": cnt, "cnt0": cnt.clone(),
            "any": case["order"] == "any", "step": 0, "f": api.Fields.per_particle()}


def _run_chi(s):
    _restore(s)
    api.qed_step_fused(s["ctx"], s["e"], s["p"], s["g"], s["f"], s["step"])
    s["step"] += 1
    out = {"e": _arrays(s["e"], STATE), "n": s["cnt"]}
    if not s["any"]:
        out["g"] = _arrays(s["g"], STATE + ("w", "id", "alive") + FIELDS)
    return out


def _prepare_cascade(case, seed):
    n, dims = case["n"], (case["nx"], case["ny"], case["nz"])
    cap, cap_g = n + n // 2 + 4096, 5 * n + 4096
    ctx = _context(dt=0.1, seed=_seed_of(case), append_order=int(case["order"] == "any"), max_particles=max(cap_g, 1 << 16))
    r = _Rand(seed)
    (e, eb), (p, pb) = _species(cap, -1, rows=STATE), _species(cap, 1, rows=STATE)
    g, gb = _species(cap_g, 0, rows=STATE[:3])
    cnt = _counts(e, p, g)
    for s, m, photon in ((e, n, False), (p, n, False), (g, 2 * n, True)):
        gam = r.log_uniform(m, 10.0, 2000.0)
        mom = (gam if photon else torch.sqrt(gam * gam - 1.0)) * r.iso(m)
        pos = (r.uniform(m, d * 0.375 * GRID_DX, d * 0.625 * GRID_DX) for d in dims)
        _fill(s, m, **_vec(STATE[:3], pos), **_vec(STATE[3:], mom), w=torch.ones(m, device="cuda"), id=_ids(r, m))
    grid = torch.zeros((case["nz"], case["ny"], case["nx"], 8), dtype=torch.float32, device="cuda")
    return {"ctx": ctx, "e": e, "p": p, "g": g, "bufs": [(b, b.clone()) for b in (eb, pb, gb)],
            "alive0": g.alive[:2 * n].clone(), "cnt": cnt, "cnt0": cnt.clone(), "n": n, "grid": grid,
            "any": case["order"] == "any", "step": 0, "f": api.Fields.grid(grid, GRID_DX, GRID_DX, GRID_DX)}


def _run_cascade(s):
    for b, b0 in s["bufs"]:
        b.copy_(b0)
    s["cnt"].copy_(s["cnt0"])
    s["g"].alive[:2 * s["n"]].copy_(s["alive0"])
    api.qed_fill_standing_wave(s["ctx"], s["grid"], 0.0, GRID_DX, 800.0, 0.1 * s["step"])
    api.qed_step_fused(s["ctx"], s["e"], s["p"], s["g"], s["f"], s["step"])
    s["step"] += 1
    kept = STATE + ("w", "id")
    g = _arrays(s["g"], STATE[:3] + ("alive",) if s["any"] else kept + ("alive",))
    if s["any"]:
        g = {k: v[:2 * s["n"]] for k, v in g.items()}
    return {"e": _arrays(s["e"], kept), "p": _arrays(s["p"], kept), "g": g, "n": s["cnt"], "grid": s["grid"]}


def _pic_inputs(case, seed):
    dims, n = (case["nx"], case["ny"], case["nz"]), case["nx"] * case["ny"] * case["nz"] * case["ppc"]
    r = _Rand(seed)
    pos = [r.uniform(n) * (d * PIC_DX) for d in dims]
    if case["cell_order"]:
        c = [torch.floor(pos[a].double() / PIC_DX).to(torch.int64) for a in range(3)]
        o = torch.argsort((c[2] * dims[1] + c[1]) * dims[0] + c[0])
        pos = [q[o] for q in pos]
    mom = [PIC_P_TH * r.normal(n) for _ in range(3)]
    w = torch.full((n,), PIC_DENSITY * PIC_DX ** 3 / case["ppc"], device="cuda")
    return dims, n, pos, mom, w, _ids(r, n)


def _prepare_pic(case, seed):
    dims, n, pos, mom, w, ids = _pic_inputs(case, seed)
    ctx = _context(dt=PIC_DT, seed=_seed_of(case), max_particles=max(n, 1 << 16))
    e = api.Species.empty(n, -1)
    _fill(e, n, **_vec(STATE, pos + mom), w=w, id=ids)
    y = api.Yee(*dims, PIC_DX, PIC_DX, PIC_DX)
    api.qed_pic_fields(ctx, y, advance=False)
    return {"ctx": ctx, "e": e, "p": api.Species.empty(0, 1), "g": api.Species.empty(1 << 16, 0), "y": y, "step": 0}


def _run_pic(s):
    api.qed_pic_step(s["ctx"], s["e"], s["p"], s["g"], s["y"], 1.0, s["step"])
    s["step"] += 1
    y = s["y"]
    return {"e": _arrays(s["e"], STATE), "y": {k: getattr(y, k) for k in FIELDS + ("nodes",)}}


def _run_sizes(case):
    """Sizes of the runs, spread over the logarithm of [lo, hi]."""
    k, lo, hi = case["runs"], case["lo"], case["hi"]
    return [int(lo * (hi / lo) ** (((37 * i) % k + 0.5) / k)) for i in range(k)]


def _prepare_batched(case, seed):
    sizes = _run_sizes(case)
    n, k = sum(sizes), case["runs"]
    cap_g = int(0.3 * n * case["steps"]) + 4096
    r = _Rand(seed)
    e, buf = _species(2 * n, -1, fields=True, tag=True)
    p = api.Species.empty(n, 1, fields=True, tag=True)
    g = api.Species.empty(cap_g, 0, fields=True, tag=True)
    cnt = _counts(e, p, g)
    tag = torch.repeat_interleave(torch.arange(k, device="cuda"), torch.tensor(sizes, device="cuda"))
    lim = torch.sort(r.log_uniform((k, 2), 0.01, 10.0), dim=1).values
    mom, b = _chi_particles(r, n, lim[tag, 0], lim[tag, 1])
    _fill(e, n, **_vec(STATE[3:], mom), **_vec(FIELDS[3:], b), w=torch.ones(n, device="cuda"), id=_ids(r, n), tag=tag)
    # the captured graph belongs to the context, so a set of runs has its own
    ctx = _new_context(dt=DT, seed=_seed_of(case), append_order=1, max_particles=max(2 * n, cap_g))
    return {"ctx": ctx, "e": e, "p": p, "g": g, "buf": buf, "buf0": buf.clone(), "cnt": cnt, "cnt0": cnt.clone(),
            "steps": case["steps"], "runs": k, "step": 0, "f": api.Fields.per_particle()}


def _run_batched(s):
    _restore(s)
    runs = api.qed_run_batched(s["ctx"], s["e"], s["p"], s["g"], s["f"], s["step"], s["steps"], n_runs=s["runs"])
    s["step"] += s["steps"]
    # pairs come from photons, whose order is free: the electrons that were there
    n = s["e"].capacity // 2
    return {"e": {k: v[:n] for k, v in _arrays(s["e"], STATE).items()}, "n": s["cnt"], "runs": runs}


def _prepare_host(case, seed):
    n = case["n"]
    cap_g = int(0.1 * n) + 4096
    ctx = _context(dt=DT, seed=_seed_of(case), max_particles=max(cap_g, case["chunk"], 1 << 16))
    r = _Rand(seed)
    h = api.Species.empty(n, -1, fields=True, pinned=True)
    g = api.Species.empty(cap_g, 0, fields=True)
    gh = api.Species.empty(cap_g, 0, fields=True, pinned=True)
    # chi up to 0.3: the ensemble, which lives on the host and is not put back, cools slowly
    mom, b = _chi_particles(r, n, 1e-3, 0.3)
    _fill(h, n, **_vec(STATE[3:], mom), **_vec(FIELDS[3:], b), w=torch.ones(n), id=_ids(r, n))
    return {"ctx": ctx, "h": h, "g": g, "gh": gh, "chunk": case["chunk"], "step": 0, "f": api.Fields.per_particle()}


def _run_host(s):
    s["g"].n.zero_()
    api.qed_lepton_step_host(s["ctx"], s["h"], s["g"], s["gh"], s["f"], s["step"], s["chunk"])
    s["step"] += 1
    return {"h": _arrays(s["h"], STATE), "gh": _arrays(s["gh"], STATE + ("w", "id") + FIELDS), "n": s["gh"].n}


def _compact_inputs(case, seed):
    n, r = case["n"], _Rand(seed)
    dtype = torch.float64 if case["precision"] == 64 else torch.float32
    arrays = {k: r.uniform(n, -1e3, 1e3, dtype) for k in STATE + ("w",) + (FIELDS if case["fields"] else ())}
    return arrays, _ids(r, n), r.uniform(n) >= case["dead"], dtype


def _prepare_compact(case, seed):
    n = case["n"]
    arrays, ids, alive, dtype = _compact_inputs(case, seed)
    ctx = _context(dt=DT, seed=_seed_of(case), precision=int(case["precision"] == 64), max_particles=max(n, 1 << 16))
    g = api.Species.empty(n, 0, dtype=dtype, fields=case["fields"])
    _fill(g, n, id=ids, **arrays)
    g.alive.copy_(alive)
    return {"ctx": ctx, "g": g, "alive0": g.alive.clone(), "n0": g.n.clone()}


def _run_compact(s):
    s["g"].alive.copy_(s["alive0"])
    s["g"].n.copy_(s["n0"])
    api.qed_compact(s["ctx"], s["g"])
    return {"g": _arrays(s["g"], STATE + ("w", "id", "alive") + FIELDS), "n": s["g"].n}


def _prepare_train(case, seed):
    ctx = _context(dt=DT, seed=_seed_of(case), sampler=1, max_particles=1 << 16)
    return {"ctx": ctx, "w": api.mlp_init_params(seed), "seed": seed, "samples": case["samples"]}


def _run_train(s):
    api.qed_mlp_load(s["ctx"], s["w"])
    loss = api.qed_mlp_train(s["ctx"], s["samples"], seed=s["seed"])
    return {"loss": loss, "w": api.qed_mlp_get(s["ctx"])}


_PREPARE = {"uniform": _prepare_uniform, "ensemble": _prepare_ensemble, "chi": _prepare_chi,
            "cascade": _prepare_cascade, "pic": _prepare_pic, "batched": _prepare_batched, "host": _prepare_host,
            "compact": _prepare_compact, "train": _prepare_train}
_RUN = {"uniform": _run_uniform, "ensemble": _run_ensemble, "chi": _run_chi, "cascade": _run_cascade,
        "pic": _run_pic, "batched": _run_batched, "host": _run_host, "compact": _run_compact, "train": _run_train}


def prepare(case, seed):
    return {"run": _RUN[case["kind"]], **_PREPARE[case["kind"]](case, seed)}


def run(state):
    return state["run"](state)


# ---- floors -----------------------------------------------------------------
def work(case):
    """Bytes: per lepton x, y, z, p, w, id (and its fields) read, x, y, z, p
    written; per photon the same without the momentum written; per new
    particle its state, id, alive flag and fields written.  The mean numbers of
    new photons per lepton and step are those of the ensembles."""
    kind = case["kind"]
    if kind == "uniform":
        w = case["precision"] // 8
        n = case["n"]
        return {"bytes": n * (13 * w + 8) + 0.014 * n * (7 * w + 9), "flops": 400.0 * n}
    if kind == "ensemble":
        return {"bytes": case["n"] * (84 + 68 + 0.1 * 61 + 0.01 * 123), "flops": 800.0 * case["n"]}
    if kind == "chi":
        n = case["n"]
        net = 2.0 * 8577 * 0.05 * n if case["sampler"] == "mlp" else 0.0
        return {"bytes": n * (84 + 0.184 * 61), "flops": 900.0 * n + net}
    if kind == "cascade":
        n = case["n"]
        return {"bytes": 2 * n * (60 + 0.5 * 37) + 2 * n * 44 + 2 * 32 * case["nx"] * case["ny"] * case["nz"],
                "flops": 5000.0 * n}
    if kind == "pic":
        cells = case["nx"] * case["ny"] * case["nz"]
        n = cells * case["ppc"]
        # the step and the deposit in one visit of a particle; E, B read and written, the nodes
        # written and read
        return {"bytes": n * 60 + cells * (48 + 64), "flops": 500.0 * n + 60.0 * cells}
    if kind == "batched":
        n = sum(_run_sizes(case))
        return {"bytes": case["steps"] * n * (84 + 0.1 * 61), "flops": case["steps"] * 600.0 * n}
    if kind == "host":
        return {"bytes": case["n"] * (84 + 0.01 * 61), "flops": 400.0 * case["n"]}
    if kind == "compact":
        n, w = case["n"], case["precision"] // 8
        rec = w * (13 if case["fields"] else 7) + 8
        return {"bytes": n * (1 + 2 * rec * (1 - case["dead"])), "flops": float(n)}
    return {"bytes": 8577 * 4 * 2, "flops": 3 * 2.0 * 8577 * case["samples"]}


# ---- 64-bit values ----------------------------------------------------------
def _boris64(p, E, B, q, dt):
    h = 0.5 * q * dt
    u = [p[c] + h * E[c] for c in range(3)]
    ig = h / torch.sqrt(1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    t = [B[c] * ig for c in range(3)]
    s2 = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    v = [u[c] + w for c, w in enumerate(cross(u, t))]
    u = [u[c] + w * s2 for c, w in enumerate(cross(v, t))]
    return [u[c] + h * E[c] for c in range(3)]


def _drift64(x, p, dt):
    g = torch.sqrt(1.0 + p[0] ** 2 + p[1] ** 2 + p[2] ** 2)
    return [x[c] + dt * p[c] / g for c in range(3)]


def _moved64(s, q, dt, B=None):
    """Positions of a species after the push (the recoil does not move it)."""
    d = {k: getattr(s, k).double() for k in STATE + (FIELDS if B is None else ())}
    p = [d[k] for k in STATE[3:]]
    E = [0.0] * 3 if B is not None else [d[k] for k in FIELDS[:3]]
    p = _boris64(p, E, B if B is not None else [d[k] for k in FIELDS[3:]], q, dt)
    return _vec(STATE[:3], _drift64([d[k] for k in STATE[:3]], p, dt))


def _weights(f, n):
    i = torch.floor(f)
    w, i = f - i, i.to(torch.int64) % n
    return (i, (i + 1) % n), (1.0 - w, w)


def _corners(frac, dims):
    ax = [_weights(frac[a], dims[a]) for a in range(3)]
    for k in range(2):
        for j in range(2):
            for i in range(2):
                yield ((ax[2][0][k] * dims[1] + ax[1][0][j]) * dims[0] + ax[0][0][i],
                       ax[0][1][i] * ax[1][1][j] * ax[2][1][k])


def _exact_pic(case, seed):
    """One cycle from fields at rest: drift, CIC current at the staggered
    positions, the leapfrog and the node means (periodic)."""
    dims, n, pos, mom, w, _ = _pic_inputs(case, seed)
    pos, mom, w = [v.double() for v in pos], [v.double() for v in mom], w.double()
    new = _drift64(pos, mom, PIC_DT)
    g = torch.sqrt(1.0 + mom[0] ** 2 + mom[1] ** 2 + mom[2] ** 2)
    J = []
    for a in range(3):
        frac = [(new[c] - 0.5 * PIC_DT * mom[c] / g) / PIC_DX - (0.5 if c == a else 0.0) for c in range(3)]
        amount = -w / PIC_DX ** 3 * mom[a] / g
        j = torch.zeros(dims[0] * dims[1] * dims[2], dtype=torch.float64, device="cuda")
        for idx, weight in _corners(frac, dims):
            j.index_add_(0, idx, amount * weight)
        J.append(j.view(dims[2], dims[1], dims[0]))
    E = [-PIC_DT * j for j in J]  # from E = B = 0: B is still 0 at the E step

    def fwd(v, a):
        return (torch.roll(v, -1, 2 - a) - v) / PIC_DX

    B = [-0.5 * PIC_DT * (fwd(E[(a + 2) % 3], (a + 1) % 3) - fwd(E[(a + 1) % 3], (a + 2) % 3)) for a in range(3)]

    def mean(v, a):
        return 0.5 * (v + torch.roll(v, 1, 2 - a))

    nodes = torch.zeros(tuple(E[0].shape) + (8,), dtype=torch.float64, device="cuda")
    for a in range(3):
        nodes[..., a] = mean(E[a], a)
        nodes[..., 3 + a] = mean(mean(B[a], (a + 1) % 3), (a + 2) % 3)
    return {"e": _vec(STATE, new + mom), "y": {**_vec(FIELDS, E + B), "nodes": nodes}}


def exact(case, seed):
    """The outputs that plain arithmetic gives: positions after the push, the
    whole PIC cycle (its plasma does not radiate) and the compaction.  Recoiled
    momenta and new particles need the quadrature of the rates per particle
    and are left out."""
    kind = case["kind"]
    if kind == "pic":
        return _exact_pic(case, seed)
    if kind == "compact":
        arrays, ids, alive, dtype = _compact_inputs(case, seed)
        out = {}
        for k, v in arrays.items():
            kept = v[alive]
            out[k] = torch.cat([kept, v[kept.numel():]]).double()
        return {"g": out, "n": None}
    if kind in ("uniform", "chi"):
        s = prepare(case, seed)
        B = [0.0, 0.0, 410.0] if kind == "uniform" else None
        return {"e": _moved64(s["e"], -1.0, DT, B)}
    if kind == "host":
        return {"h": _moved64(prepare(case, seed)["h"], -1.0, DT)}
    return None
