"""Timed cases of the Vlasov-Hybrid library: what one pass is, its inputs, the
work it cannot do without, and its result in plain FP64 torch.

A case is a dict of plain values; its "kind" says which call a user makes:

step     one context: a few time steps, then the state a run writes out (f and
         n of every species, rho, E, the diagnostics row)
batch    many small runs advanced together, then f, n, rho and E of every run
adjoint  the field energy at the end of a run and its gradient
load     markers of a saved state into a context, then the state as above
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _step1(name, precision, nx, nv, px, pv, f0, steps, ions=False, softening=True, L=0.0, vmax=6.0, dt=0.1):
    c = dict(kind="step", nvdim=1, precision=precision, nx=nx, nv=nv, px=px, pv=pv, f0=f0, steps=steps, ions=ions,
             softening=softening, L=L, vmax=vmax, dt=dt)
    return dict(c, name=name) if name else c


def _step3(name, precision, nx, nvx, nvy, nvz, px, pv, f0, steps, L, vmax=8.0, dt=0.05, bx=0.0, by=0.0, bz=0.0):
    c = dict(kind="step", nvdim=3, precision=precision, nx=nx, nvx=nvx, nvy=nvy, nvz=nvz, px=px, pv=pv, f0=f0,
             steps=steps, softening=True, L=L, vmax=vmax, dt=dt, bx=bx, by=by, bz=bz)
    return dict(c, name=name) if name else c


def listed():
    bump_L = 2 * math.pi / 0.3
    return [
        # the smallest production run: Landau damping at k = 0.5, 32768
        # markers, FP64; every kernel is short, so latency and launches count
        _step1("landau 64x128 fp64", "fp64", 64, 128, 2, 2, "landau", 20, L=4 * math.pi),
        # a grid that is no power of two, odd in velocity, nine markers per
        # cell: a user's own parameter study in the fast precision
        _step1("ragged 300x333 fp32", "fp32", 300, 333, 3, 3, "two_stream", 8, L=120.0, vmax=10.0, dt=0.05,
               softening=False),
        # two-stream instability with mobile ions, 16.8 M markers, FP32
        _step1("two-stream 512x1024 fp32", "fp32", 512, 1024, 4, 4, "two_stream", 4, ions=True, L=204.8, vmax=10.0,
               dt=0.05),
        # the paper's own Landau run at its production size, FP64
        _step1("landau paper 512x6600 fp64", "fp64", 512, 6600, 2, 2, "landau", 2, L=5 * math.pi, vmax=10.0),
        # bump-on-tail 1d3v, 134 M markers: the largest run, in the paper's
        # precision and in the fast one
        _step3("bump 256x64^3 fp64", "fp64", 256, 64, 64, 64, 2, 1, "bump", 1, bump_L),
        _step3("bump 256x64^3 fp32", "fp32", 256, 64, 64, 64, 2, 1, "bump", 1, bump_L),
        # electron Bernstein geometry: a uniform field across x, Boris push
        _step3("bernstein 256x64^3 fp32", "fp32", 256, 64, 64, 64, 2, 1, "bernstein", 1, 128.0, vmax=6.0, dt=0.1,
               bz=1.0),
        # a small odd 1d3v grid with an oblique field, FP64
        _step3("oblique 100x24x20x18 fp64", "fp64", 100, 24, 20, 18, 3, 1, "bernstein", 4, 50.0, vmax=5.0, dt=0.1,
               bx=0.3, by=-0.9, bz=1.4),
        # a parameter study: 64 small runs of mixed sizes advanced together
        dict(name="ensemble of 64 fp32", kind="batch", precision="fp32", nrun=64, steps=10),
        # gradient of the final field energy (inverse problems), both precisions
        dict(name="adjoint 256x512 fp32", kind="adjoint", precision="fp32", nx=256, nv=512, px=2, pv=4, nmode=16,
             steps=100, ckpt=25, L=102.4),
        dict(name="adjoint 256x512 fp64", kind="adjoint", precision="fp64", nx=256, nv=512, px=2, pv=4, nmode=16,
             steps=100, ckpt=25, L=102.4),
        # restart: the markers of a saved 1d3v state, 16.8 M of them
        dict(name="restart 256x32^3 fp64", kind="load", nvdim=3, precision="fp64", nx=256, nvx=32, nvy=32, nvz=32,
             npc=2, L=bump_L, vmax=8.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """A grid size: half of them powers of two, the others anything."""
    n = _log_int(rng, lo, hi)
    return 1 << max(2, int(round(math.log2(n)))) if rng.random() < 0.5 else n


def draw(rng):
    prec = rng.choice(["fp32", "fp64"])
    kind = rng.choices(["step1", "step3", "adjoint", "load", "batch"], [6, 6, 2, 2, 1])[0]
    if kind == "step1":
        nx, nv = _grid(rng, 24, 900), _log_int(rng, 64, 6600)
        px, pv = rng.choice([(1, 2), (2, 2), (2, 4), (3, 3), (4, 4)])
        while nx * nv * px * pv > 16e6:
            nv = max(64, nv // 2)
        f0 = rng.choice(["landau", "two_stream"])
        return _step1("", prec, nx, nv, px, pv, f0, rng.randint(1, 12), ions=rng.random() < 0.4,
                      softening=rng.random() < 0.7, L=0.4 * nx if f0 == "two_stream" else rng.uniform(10.0, 20.0),
                      vmax=10.0 if f0 == "two_stream" else rng.uniform(5.0, 10.0), dt=rng.choice([0.05, 0.1]))
    if kind == "step3":
        nx = min(_grid(rng, 12, 400), 512)
        nv = [_log_int(rng, 8, 48) for _ in range(3)]
        while nx * nv[0] * nv[1] * nv[2] > 8e6:
            nv[rng.randrange(3)] = 8
        px, pv = rng.choice([(1, 1), (2, 1), (3, 1), (2, 2)])
        f0 = rng.choice(["bump", "bernstein"])
        b = [rng.uniform(-1.5, 1.5) for _ in range(3)] if f0 == "bernstein" else [0.0] * 3
        return _step3("", prec, nx, nv[0], nv[1], nv[2], px, pv, f0, rng.randint(1, 6), rng.uniform(0.08, 0.5) * nx,
                      vmax=rng.uniform(5.0, 8.0), dt=rng.choice([0.05, 0.1]), bx=b[0], by=b[1], bz=b[2])
    if kind == "adjoint":
        nx, steps = _grid(rng, 32, 400), rng.randint(10, 80)
        return dict(kind="adjoint", precision=prec, nx=nx, nv=_log_int(rng, 64, 600), px=rng.choice([1, 2]),
                    pv=rng.choice([2, 4]), nmode=rng.randint(1, 16), steps=steps, ckpt=rng.randint(5, steps),
                    L=0.4 * nx)
    if kind == "load":
        nvdim = rng.choice([1, 3])
        nx = min(_grid(rng, 24, 600), 512)
        nv = [_log_int(rng, 64, 4000), 1, 1] if nvdim == 1 else [_log_int(rng, 8, 32) for _ in range(3)]
        return dict(kind="load", nvdim=nvdim, precision=prec, nx=nx, nvx=nv[0], nvy=nv[1], nvz=nv[2],
                    npc=rng.choice([1, 2, 3]), L=0.1 * nx, vmax=rng.uniform(5.0, 8.0))
    return dict(kind="batch", precision=prec, nrun=rng.randint(8, 48), steps=rng.randint(2, 10))


# ---------------------------------------------------------------------------
# what the program of a case knows: domain, species, f0, lattice, seeds
# ---------------------------------------------------------------------------
def _beam(n, u, vth):
    return (n, (u, 0.0, 0.0), (vth, 1.0, 1.0))


def _modes(rng, k, amp):
    return [(m + 1, amp * rng.uniform(0.5, 1.5), rng.uniform(0.0, 2 * math.pi)) for m in range(k)]


def _species(q, m, nv, vmin, vmax, mobile=True):
    return dict(q=q, m=m, nv=list(nv), vmin=list(vmin), vmax=list(vmax), mobile=mobile)


def _problem(case, seed):
    """A run as plain values: its domain, species, initial distributions."""
    rng = random.Random(seed * 1000003 + 17)
    p = dict(nvdim=case.get("nvdim", 1), nx=case["nx"], L=case["L"], dt=case.get("dt", 0.05), cP=1.0,
             softening=case.get("softening", True), precision=case["precision"], seed=rng.getrandbits(48), jitter=1.0,
             B=[case.get(k, 0.0) for k in ("bx", "by", "bz")])
    if p["nvdim"] == 3:
        v = case["vmax"]
        p["species"] = [_species(-1.0, 1.0, [case["nvx"], case["nvy"], case["nvz"]], [-v] * 3, [v] * 3)]
        if case.get("f0", "bump") == "bump":
            beams = [(0.95, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)), (0.05, (4.0, 0.0, 0.0), (0.5, 0.5, 0.5))]
            p["f0"] = [(beams, _modes(rng, 1, 1e-3))]
        else:
            p["f0"] = [([(1.0, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0))], _modes(rng, 4, 1e-3))]
        p["lattice"] = [[case.get("px", 1), case.get("pv", 1), 1, 1]]
        return p
    v = case.get("vmax", 10.0)
    p["species"] = [_species(-1.0, 1.0, [case["nv"] if "nv" in case else case["nvx"]], [-v], [v])]
    if case.get("f0", "two_stream") == "landau":
        p["f0"] = [([_beam(1.0, 0.0, 1.0)], [(1, 0.05 * rng.uniform(0.5, 1.5), rng.uniform(0.0, 2 * math.pi))])]
    else:
        nmode = case.get("nmode", min(8, case["nx"] // 8))
        p["f0"] = [([_beam(0.5, 3.0, 1.0), _beam(0.5, -3.0, 1.0)], _modes(rng, nmode, 1e-3))]
    p["lattice"] = [[case.get("px", 1), case.get("pv", 1), 1, 1]]
    if case.get("ions"):
        vt = 1836.0 ** -0.5
        p["species"].append(_species(1.0, 1836.0, p["species"][0]["nv"], [-10.0 * vt], [10.0 * vt]))
        p["f0"].append(([_beam(1.0, 0.0, vt)], []))
        p["lattice"].append(p["lattice"][0])
    return p


def _ensemble(case, seed):
    """nrun small 1d1v runs: Landau or two-stream, sizes drawn from the
    ensemble's own (the same sizes for every seed, other parameters)."""
    size, rng = random.Random(case["nrun"]), random.Random(seed * 1000003 + 29)
    runs = []
    for _ in range(case["nrun"]):
        landau = size.random() < 0.5
        px, pv = size.choice([(2, 2), (2, 4), (4, 4)])
        nx, nv = size.choice([64, 128, 256, 512]), size.choice([128, 256, 512, 1024])
        u, amp = rng.uniform(0.0, 4.0), math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))
        p = dict(nvdim=1, nx=nx, L=4 * math.pi if landau else 0.4 * nx, dt=0.1 if landau else 0.05, cP=1.0,
                 softening=True, precision=case["precision"], seed=rng.getrandbits(48), jitter=1.0, B=[0.0] * 3,
                 lattice=[[px, pv, 1, 1]])
        if landau:
            p["species"] = [_species(-1.0, 1.0, [nv], [u - 6.0], [u + 6.0])]
            p["f0"] = [([_beam(1.0, u, 1.0)], [(1, amp, 0.0)])]
        else:
            p["species"] = [_species(-1.0, 1.0, [nv], [-10.0], [10.0])]
            p["f0"] = [([_beam(0.5, u, 1.0), _beam(0.5, -u, 1.0)], _modes(rng, 4, amp))]
        runs.append(p)
    return runs


def _cells(p, s):
    return p["nx"] * math.prod(p["species"][s]["nv"])


def _saved_markers(case, p, seed):
    """The markers of a saved state: one velocity cell after the other (v_z,
    v_y, v_x slowest), random in x, f = f0."""
    sp, nd = p["species"][0], p["nvdim"]
    nvc = math.prod(sp["nv"])
    n = nvc * p["nx"] * case["npc"]
    # random numbers from a counter, so that they are the same on any device
    base = random.Random(seed * 1000003 + 41).getrandbits(40)
    k = torch.arange(n, device=DEV)
    cell = k // (p["nx"] * case["npc"])
    jx = cell % sp["nv"][0]
    rest = cell // sp["nv"][0]
    j = [jx] if nd == 1 else [jx, rest % sp["nv"][1], rest // sp["nv"][1]]
    x = _uniform(base, 0, k, 0) * p["L"]
    x = torch.where(x < p["L"], x, torch.zeros_like(x))
    v = torch.empty(nd, n, dtype=torch.float64, device=DEV)
    for d in range(nd):
        dv = (sp["vmax"][d] - sp["vmin"][d]) / sp["nv"][d]
        v[d] = sp["vmin"][d] + (j[d] + _uniform(base, 0, k, 1 + d)) * dv
    return x, v, _f0(p, 0, x, v)


# ---------------------------------------------------------------------------
# prepare and run: the library
# ---------------------------------------------------------------------------
def _simulation(A, p):
    prec = A.AVL_FP32 if p["precision"] == "fp32" else A.AVL_FP64
    dom = A.make_domain(p["nvdim"], p["nx"], p["L"], p["dt"], p["cP"], p["softening"], prec)
    return dom, [A.make_species(s["q"], s["m"], s["nv"], s["vmin"], s["vmax"], s["mobile"]) for s in p["species"]]


def _fill(A, sim, p):
    for s, (beams, modes) in enumerate(p["f0"]):
        sim.init_markers(s, p["lattice"][s], A.make_f0(beams, modes), p["seed"], p["jitter"])


def _outputs(p):
    """Device buffers for f and n of every species, rho, E; pinned host memory
    for the diagnostics row."""
    o = {}
    for s, sp in enumerate(p["species"]):
        shape = [p["nx"]] + sp["nv"]
        o["f%d" % s] = torch.empty(shape, dtype=torch.float64, device="cuda")
        o["n%d" % s] = torch.empty(shape, dtype=torch.float64, device="cuda")
    o["rho"] = torch.empty(p["nx"], dtype=torch.float64, device="cuda")
    o["E"] = torch.empty(p["nx"], dtype=torch.float64, device="cuda")
    o["diag"] = torch.zeros(3 + 3 * len(p["species"]), dtype=torch.float64).pin_memory()
    return o


def _read(A, ctx, o, ns):
    for s in range(ns):
        A.check(A.avl_get_f(ctx, s, o["f%d" % s].data_ptr(), o["n%d" % s].data_ptr(), 1), ctx)
    A.check(A.avl_get_rho(ctx, o["rho"].data_ptr(), 1), ctx)
    A.check(A.avl_get_E(ctx, o["E"].data_ptr(), 1), ctx)


def prepare(case, seed):
    from paper_1804_03901_gb300 import avl as A
    stream = torch.cuda.Stream()
    st = dict(case=case, A=A, stream=stream)
    if case["kind"] == "batch":
        st["p"] = runs = _ensemble(case, seed)
        made = [_simulation(A, p) for p in runs]
        b = st["batch"] = A.Batch([m[0] for m in made], [m[1] for m in made], stream.cuda_stream)
        for v, p in zip(b.runs, runs):
            _fill(A, v, p)
        # one buffer per quantity, run after run
        st["at"] = np.concatenate([[0], np.cumsum([_cells(p, 0) for p in runs])]).tolist()
        st["xat"] = np.concatenate([[0], np.cumsum([p["nx"] for p in runs])]).tolist()
        st["out"] = {k: torch.empty(st["at"][-1] if k in "fn" else st["xat"][-1], dtype=torch.float64, device="cuda")
                     for k in ("f", "n", "rho", "E")}
        return st
    st["p"] = p = _problem(case, seed)
    dom, species = _simulation(A, p)
    sim = st["sim"] = A.Simulation(dom, species, stream.cuda_stream)
    if case["kind"] == "load":
        st["out"], st["markers"] = _outputs(p), _saved_markers(case, p, seed)
        return st
    if case["kind"] == "step":
        _fill(A, sim, p)
        if any(p["B"]):
            sim.set_bfield(p["B"])
        st["out"] = _outputs(p)
        return st
    _fill(A, sim, p)
    st["theta"] = A.make_f0(*p["f0"][0])
    return st


def run(state):
    case, A = state["case"], state["A"]
    if case["kind"] == "adjoint":
        J, g_amp, g_u = state["sim"].adjoint(0, state["theta"], case["steps"], case["ckpt"])
        return {"J": J, "d_amp": g_amp, "d_drift": g_u}
    o = state["out"]
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        at, xat = state["at"], state["xat"]
        for r, v in enumerate(state["batch"].runs):
            A.check(A.avl_get_f(v.ctx, 0, o["f"].data_ptr() + 8 * at[r], o["n"].data_ptr() + 8 * at[r], 1), v.ctx)
            A.check(A.avl_get_rho(v.ctx, o["rho"].data_ptr() + 8 * xat[r], 1), v.ctx)
            A.check(A.avl_get_E(v.ctx, o["E"].data_ptr() + 8 * xat[r], 1), v.ctx)
        return o
    sim = state["sim"]
    if case["kind"] == "load":
        x, v, f = state["markers"]
        sim.set_markers(0, x, v, f)
    else:
        sim.step(case["steps"])
    _read(A, sim.ctx, o, len(sim.species))
    sim.get_diag_async(o["diag"].data_ptr())
    return o


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------
def _step_work(p, steps):
    """Markers: position, velocity and value read, position and the velocity
    components that change written, every step; the grid f and n written once
    at the end.  Arithmetic: gather, push, weights, deposit per marker."""
    w = 4 if p["precision"] == "fp32" else 8
    nd = p["nvdim"]
    pos = 8                                    # FP32: cell and offset
    turned = nd if any(p["B"]) else 1
    by = fl = 0
    for s, sp in enumerate(p["species"]):
        n = _cells(p, s) * math.prod(p["lattice"][s])
        by += steps * n * (2 * pos + w * (nd + turned) + w) + 16 * _cells(p, s)
        fl += steps * (n * (33 if nd == 1 else 89) + 8 * _cells(p, s))
    return by + 16 * p["nx"], fl


def work(case):
    if case["kind"] == "batch":
        got = [_step_work(p, case["steps"]) for p in _ensemble(case, 0)]
        return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}
    p = _problem(case, 0)
    w = 4 if p["precision"] == "fp32" else 8
    if case["kind"] == "load":
        n, cells = _cells(p, 0) * case["npc"], _cells(p, 0)
        stored = 8 + w * (p["nvdim"] + 1)
        return {"bytes": n * (8 * (2 + p["nvdim"]) + stored) + 16 * cells, "flops": n * (33 if p["nvdim"] == 1 else 89)}
    if case["kind"] == "adjoint":
        # forward step; backward: state and value read, lambda and mu updated
        n, cells = _cells(p, 0) * math.prod(p["lattice"][0]), _cells(p, 0)
        fwd, bwd = 2 * (8 + w) + w, 8 + 2 * w + 2 * (2 * w + 8)
        return {"bytes": case["steps"] * (n * (fwd + bwd) + 4 * w * cells), "flops": case["steps"] * n * (33 + 60)}
    by, fl = _step_work(p, case["steps"])
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same in plain FP64 torch
# ---------------------------------------------------------------------------
def _i64(u):
    return u - (1 << 64) if u >= 1 << 63 else u


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _uniform(seed, s, m, d):
    """SplitMix64 draw of stream index (s << 48) | (4 m + d), in [0, 1)."""
    n = (4 * m + d) | (s << 48)
    z = (n + 1) * _i64(0x9E3779B97F4A7C15) + _i64(seed)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return _shr(z ^ _shr(z, 31), 11).to(torch.float64) * (1.0 / 9007199254740992.0)


def _f0(p, s, x, v, amps=None, drifts=None):
    beams, modes = p["f0"][s]
    pert = torch.ones_like(x)
    for k, (m, amp, ph) in enumerate(modes):
        pert = pert + (amp if amps is None else amps[k]) * torch.cos(2 * math.pi * m / p["L"] * x + ph)
    tot = torch.zeros_like(x)
    for b, (n, u, vth) in enumerate(beams):
        g = n
        for d in range(p["nvdim"]):
            t = (v[d] - (u[d] if d or drifts is None else drifts[b])) / vth[d]
            g = g * torch.exp(-0.5 * t * t) / (math.sqrt(2 * math.pi) * vth[d])
        tot = tot + g
    return tot * pert


def _lattice(p, s):
    """Creation lattice: x in cells, v, in marker order (row-major cells)."""
    sp, nd = p["species"][s], p["nvdim"]
    lat, nv = p["lattice"][s][:1 + nd], sp["nv"]
    ppc, n = math.prod(lat), _cells(p, s) * math.prod(lat)
    xi = torch.empty(n, dtype=torch.float64, device=DEV)
    v = torch.empty(nd, n, dtype=torch.float64, device=DEV)
    for a in range(0, n, 1 << 24):
        m = torch.arange(a, min(n, a + (1 << 24)), device=DEV)
        cell, sub = m // ppc, m % ppc
        idx, sb = [], []
        for d in reversed(range(nd)):
            idx.insert(0, cell % nv[d])
            cell = cell // nv[d]
            sb.insert(0, sub % lat[1 + d])
            sub = sub // lat[1 + d]
        J = [(_uniform(p["seed"], s, m, d) - 0.5) * p["jitter"] for d in range(1 + nd)]
        xi[a:a + m.numel()] = cell + (sub + 0.5 + J[0]) / lat[0]
        for d in range(nd):
            dv = (sp["vmax"][d] - sp["vmin"][d]) / nv[d]
            v[d, a:a + m.numel()] = sp["vmin"][d] + (idx[d] + (sb[d] + 0.5 + J[1 + d]) / lat[1 + d]) * dv
    return xi, v


def _cic(t):
    fl = torch.floor(t - 0.5)
    return fl.to(torch.int64), t - 0.5 - fl


def _poisson(p, rho):
    nx, dx = p["nx"], p["L"] / p["nx"]
    h = torch.fft.rfft(rho)
    k = 2 * math.pi / p["L"] * torch.arange(h.numel(), dtype=torch.float64, device=rho.device)
    kappa, K2 = (torch.sin(k * dx) / dx, (2 * torch.sin(0.5 * k * dx) / dx) ** 2) if p["softening"] else (k, k * k)
    g = torch.zeros_like(k)
    last = h.numel() - 1 if nx % 2 == 0 else h.numel()
    g[1:last] = p["cP"] * kappa[1:last] / K2[1:last]
    return torch.fft.irfft(-1j * g * h, n=nx)


def _weights(p, s, xi, v):
    """(cell index [x][v...], weight) of the cloud-in-cell corners."""
    sp, nd = p["species"][s], p["nvdim"]
    i0, u = _cic(xi)
    axes = [((i0 % p["nx"], 1 - u), ((i0 + 1) % p["nx"], u))]
    for d in range(nd):
        n, dv = sp["nv"][d], (sp["vmax"][d] - sp["vmin"][d]) / sp["nv"][d]
        j0, w = _cic((v[d] - sp["vmin"][d]) / dv)
        axes.append([(j.clamp(0, n - 1), torch.where((j >= 0) & (j < n), a, torch.zeros_like(a)))
                     for j, a in ((j0, 1 - w), (j0 + 1, w))])
    for c in range(1 << (1 + nd)):
        idx, wt = axes[0][c & 1]
        for d in range(nd):
            j, a = axes[1 + d][(c >> (1 + d)) & 1]
            idx, wt = idx * sp["nv"][d] + j, wt * a
        yield idx, wt


def _reconstruct(p, s, xi, v, f):
    num = torch.zeros(_cells(p, s), dtype=torch.float64, device=xi.device)
    den = torch.zeros_like(num)
    step = 1 << 23
    for a in range(0, xi.numel(), step):
        sl = slice(a, a + step)
        for idx, wt in _weights(p, s, xi[sl], v[:, sl]):
            num = num.index_add(0, idx, wt * f[sl]) if num.requires_grad or wt.requires_grad or f.requires_grad \
                else num.index_add_(0, idx, wt * f[sl])
            den = den.index_add(0, idx, wt) if den.requires_grad or wt.requires_grad else den.index_add_(0, idx, wt)
    has = den > 0
    return torch.where(has, num / torch.where(has, den, torch.ones_like(den)), torch.zeros_like(num)), den


def _charge(p, s, f):
    sp = p["species"][s]
    dvol = math.prod((sp["vmax"][d] - sp["vmin"][d]) / sp["nv"][d] for d in range(p["nvdim"]))
    return sp["q"] * dvol * f.reshape(p["nx"], -1).sum(1)


def _push(p, s, xi, v, E):
    """New (x in cells, v) after one step in the field E."""
    sp, nx = p["species"][s], p["nx"]
    i0, u = _cic(xi)
    El = (1 - u) * E.index_select(0, i0 % nx) + u * E.index_select(0, (i0 + 1) % nx)
    qm, dt = sp["q"] / sp["m"], p["dt"]
    if p["nvdim"] == 3 and any(p["B"]):
        a = 0.5 * qm * dt
        t = [a * b for b in p["B"]]
        t2 = sum(b * b for b in t)
        sv = [2 * b / (1 + t2) for b in t]
        m = [v[0] + a * El, v[1], v[2]]
        q = [m[k] + m[(k + 1) % 3] * t[(k + 2) % 3] - m[(k + 2) % 3] * t[(k + 1) % 3] for k in range(3)]
        v = [m[k] + q[(k + 1) % 3] * sv[(k + 2) % 3] - q[(k + 2) % 3] * sv[(k + 1) % 3] for k in range(3)]
        v = torch.stack([v[0] + a * El, v[1], v[2]])
    else:
        v = torch.cat([(v[0] + qm * dt * El)[None], v[1:]])
    return torch.remainder(xi + v[0] * (dt * nx / p["L"]), nx), v


def _diag(p, fs, E):
    per = []
    for s, f in enumerate(fs):
        sp = p["species"][s]
        dv = [(sp["vmax"][d] - sp["vmin"][d]) / sp["nv"][d] for d in range(p["nvdim"])]
        v2 = torch.zeros([1] * p["nvdim"], dtype=torch.float64, device=f.device)
        for d in range(p["nvdim"]):
            c = sp["vmin"][d] + (torch.arange(sp["nv"][d], dtype=torch.float64, device=f.device) + 0.5) * dv[d]
            v2 = v2 + (c * c).reshape([-1 if e == d else 1 for e in range(p["nvdim"])])
        fx = f.reshape(p["nx"], -1)
        cell = math.prod(dv) * p["L"] / p["nx"]
        ent = torch.where(fx > 0, fx * torch.log(torch.where(fx > 0, fx, torch.ones_like(fx))), torch.zeros_like(fx))
        per.append((0.5 * sp["m"] * float((fx * v2.reshape(1, -1)).sum()) * cell, float(fx.sum()) * cell,
                    float(ent.sum()) * cell))
    we = float((E * E).sum()) * p["L"] / p["nx"] / (2 * p["cP"])
    wk = sum(q[0] for q in per)
    return torch.tensor([we, wk, we + wk] + [q[k] for k in range(3) for q in per], dtype=torch.float64)


def _state(p, fs, ns, rho, E):
    o = {}
    for s, sp in enumerate(p["species"]):
        shape = [p["nx"]] + sp["nv"]
        o["f%d" % s], o["n%d" % s] = fs[s].reshape(shape), ns[s].reshape(shape)
    return dict(o, rho=rho, E=E, diag=_diag(p, fs, E))


def _advance(p, marks, steps):
    """State after `steps` steps of the markers [(x in cells, v, f)]."""
    fs, ns = [None] * len(marks), [None] * len(marks)
    E = rho = None
    for k in range(steps + 1):
        for s, (xi, v, f) in enumerate(marks):
            if k:
                for a in range(0, xi.numel(), 1 << 23):
                    sl = slice(a, a + (1 << 23))
                    xi[sl], v[:, sl] = _push(p, s, xi[sl], v[:, sl], E)
            fs[s], ns[s] = _reconstruct(p, s, xi, v, f)
        rho = sum(_charge(p, s, f) for s, f in enumerate(fs))
        E = _poisson(p, rho)
    return _state(p, fs, ns, rho, E)


def _create(p, s):
    xi, v = _lattice(p, s)
    f = torch.empty_like(xi)
    for a in range(0, xi.numel(), 1 << 23):
        sl = slice(a, a + (1 << 23))
        f[sl] = _f0(p, s, xi[sl] * (p["L"] / p["nx"]), v[:, sl])
    return xi, v, f


def _energy_gradient(case, p):
    from torch.utils.checkpoint import checkpoint
    amps = torch.tensor([m[1] for m in p["f0"][0][1]], dtype=torch.float64, device=DEV, requires_grad=True)
    drifts = torch.tensor([b[1][0] for b in p["f0"][0][0]], dtype=torch.float64, device=DEV, requires_grad=True)
    xi, v = _lattice(p, 0)
    f = _f0(p, 0, xi * (p["L"] / p["nx"]), v, amps, drifts)

    def field(xi, v):
        return _poisson(p, _charge(p, 0, _reconstruct(p, 0, xi, v, f)[0]))

    for _ in range(case["steps"]):
        xi, v = checkpoint(lambda a, b: _push(p, 0, a, b, field(a, b)), xi, v, use_reentrant=False)
    E = field(xi, v)
    J = 0.5 * (E * E).sum() * (p["L"] / p["nx"])
    g = torch.autograd.grad(J, [amps, drifts])
    return {"J": float(J.detach()), "d_amp": g[0].detach().cpu(), "d_drift": g[1].detach().cpu()}


def exact(case, seed):
    if case["kind"] == "batch":
        got = [_advance(p, [_create(p, 0)], case["steps"]) for p in _ensemble(case, seed)]
        return {k: torch.cat([g[a].reshape(-1) for g in got]) for k, a in (("f", "f0"), ("n", "n0"), ("rho", "rho"),
                                                                          ("E", "E"))}
    p = _problem(case, seed)
    if case["kind"] == "adjoint":
        return _energy_gradient(case, p)
    if case["kind"] == "load":
        x, v, f = _saved_markers(case, p, seed)
        return _advance(p, [(x / (p["L"] / p["nx"]), v, f)], 0)
    return _advance(p, [_create(p, s) for s in range(len(p["species"]))], case["steps"])
