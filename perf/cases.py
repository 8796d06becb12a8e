"""The work a user of this library has it do, as cases that can be timed.

A case is a dict of plain values; ``listed()`` gives the standing ones and
``draw()`` more of the same ranges.  Sizes come from the workload
descriptions, the tests and the benchmark of this repository: the plane wave
(256 to 4096 electrons), the 2D laser-on-foil (131072 electrons on a
2048x512 grid), the beam collision around its pulse peak, the constant-B
cascade, super-photon coalescence and the serving stream.

Every pass starts from the same state: the live slots, the live counts and
the grid are put back from a copy on the device (on the host for
``run_host``), as a program does that runs an ensemble from one checkpoint.
"""
from __future__ import annotations

import math
import random
import weakref

import numpy as np
import torch

from paper_1311_1107_gb300 import qedpic as Q
from paper_1311_1107_gb300 import workloads as W
from paper_1311_1107_gb300.serve import ServingEngine
from paper_1311_1107_gb300.sim import Simulation

DEV = "cuda:0"
ROWS3 = ("x", "y", "z", "ux", "uy", "uz", "tau", "w")
SPECIES = ("electron", "positron", "photon")


def listed() -> list:
    return [
        # a small plane-wave run, one launch a step, on the default precision:
        # the smallest call, where latency and launches count
        {"name": "plane 256 fp64", "family": "plane", "n": 256, "precision": "fp64", "steps": 20,
         "photons": 1.0},
        # the plane-wave job (4096 e-) as a fused window
        {"name": "fused 4096 mixed", "family": "fused", "n": 4096, "precision": "mixed",
         "steps": 250, "photons": 0.0},
        # the 2D foil in the fixed pulse snapshot: the benchmark's headline
        {"name": "foil mixed", "family": "foil", "ny": 512, "nx": 2048, "ppc": 8, "cells": 32,
         "precision": "mixed", "steps": 10, "fields": "fixed", "photons": 0.5, "pairs": 0.01},
        # the same on the FP64 path
        {"name": "foil fp64", "family": "foil", "ny": 512, "nx": 2048, "ppc": 8, "cells": 32,
         "precision": "fp64", "steps": 5, "fields": "fixed", "photons": 0.5, "pairs": 0.01},
        # the foil with its state in host memory, copied in and out by the call
        {"name": "foil host", "family": "host", "ny": 512, "nx": 2048, "ppc": 8, "cells": 32,
         "precision": "mixed", "steps": 2, "photons": 0.5, "pairs": 0.01},
        # the foil as a PIC cycle: sort by cell, then Yee solver, current
        # deposition and the QED step, on a grid whose rows are odd in number
        {"name": "foil pic", "family": "pic", "ny": 511, "nx": 2048, "ppc": 8, "cells": 32,
         "precision": "mixed", "steps": 8, "photons": 0.5, "pairs": 0.05},
        # the beam collision around the pulse peak, leptons first
        {"name": "collision mixed", "family": "collision", "n": 4_000_001, "precision": "mixed",
         "steps": 6, "start": 980, "positrons": 0.05, "photons": 0.5, "dead": 0.1},
        # the same on the FP64 path
        {"name": "collision fp64", "family": "collision", "n": 200_003, "precision": "fp64",
         "steps": 5, "start": 980, "positrons": 0.05, "photons": 0.5, "dead": 0.1},
        # the collision after its peak: photons outnumber the leptons, a part
        # of them has decayed
        {"name": "photons mixed", "family": "collision", "n": 1_000_000, "precision": "mixed",
         "steps": 6, "start": 1060, "positrons": 0.5, "photons": 10.0, "dead": 0.25},
        # the paper's constant-B cascade with its energy, number and mean chi
        # read as it goes (the quantities of the paper's figures)
        {"name": "cascade diag fp64", "family": "cascade", "n": 16384, "precision": "fp64",
         "steps": 5, "reads": 2, "positrons": 0.2, "photons": 4.0},
        # coalescence of the collision's super-photons on a box grid
        {"name": "coalesce", "family": "coalesce", "n": 4_000_000, "nx": 64, "ny": 32, "nz": 32,
         "energy_bins": 8, "direction_bins": 8, "min_group": 3, "dead": 0.05, "merge": True},
        # independent collision requests served in shared launches
        {"name": "serving", "family": "serving", "requests": 6, "n_min": 1000, "n_max": 100_000,
         "steps_min": 100, "steps_max": 400},
    ]


def _log(rng: random.Random, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random) -> dict:
    family = rng.choice(("plane", "fused", "foil", "foil", "host", "pic", "collision",
                         "collision", "cascade", "coalesce", "serving"))
    precision = rng.choice(("mixed", "fp64"))
    if family == "plane":
        return {"family": family, "n": int(_log(rng, 100, 20_000)), "precision": precision,
                "steps": rng.randint(5, 40), "photons": round(rng.uniform(0.0, 4.0), 3)}
    if family == "fused":
        return {"family": family, "n": int(_log(rng, 300, 20_000)), "precision": precision,
                "steps": int(_log(rng, 20, 300)), "photons": round(rng.uniform(0.0, 2.0), 3)}
    if family in ("foil", "host", "pic"):
        c = {"family": family, "ny": rng.randint(60, 560), "nx": rng.randint(500, 2100),
             "ppc": rng.randint(2, 9), "cells": rng.randint(8, 32),
             "precision": precision if family == "foil" else "mixed",
             "steps": rng.randint(2, 5) if family == "host" else rng.randint(3, 8),
             "photons": round(rng.uniform(0.0, 1.5), 3), "pairs": round(rng.uniform(0.0, 0.1), 3)}
        if family == "foil":
            c["fields"] = rng.choice(("fixed", "refill"))
        if family == "pic" and rng.random() < 0.5:
            c["nx"] = c["nx"] // 4 * 4
        return c
    if family == "collision":
        top = 3_000_000 if precision == "mixed" else 200_000
        photons = _log(rng, 0.1, 10.0)
        n = _log(rng, 2000, top / (1.0 + 0.25 * photons))
        return {"family": family, "n": int(n), "precision": precision, "steps": rng.randint(3, 6),
                "start": rng.randint(900, 1080), "positrons": round(rng.uniform(0.0, 0.5), 3),
                "photons": round(photons, 3), "dead": round(rng.uniform(0.0, 0.4), 3)}
    if family == "cascade":
        return {"family": family, "n": int(_log(rng, 500, 16_000)), "precision": precision,
                "steps": rng.randint(2, 6), "reads": rng.randint(1, 3),
                "positrons": round(rng.uniform(0.0, 0.4), 3),
                "photons": round(rng.uniform(0.5, 5.0), 3)}
    if family == "coalesce":
        return {"family": family, "n": int(_log(rng, 20_000, 4_000_000)),
                "nx": rng.randint(8, 80), "ny": rng.randint(4, 40), "nz": rng.randint(4, 40),
                "energy_bins": rng.choice((4, 8, 16)), "direction_bins": rng.choice((4, 8, 16)),
                "min_group": rng.randint(3, 6), "dead": round(rng.uniform(0.0, 0.5), 3),
                "merge": rng.random() < 0.75}
    return {"family": "serving", "requests": rng.randint(2, 6), "n_min": 1000,
            "n_max": int(_log(rng, 3000, 100_000)), "steps_min": 50,
            "steps_max": rng.randint(60, 400)}


# ---------------------------------------------------------------- populations

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _unit(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _depths(g, n: int):
    return -torch.log1p(-_unit(g, n))


def _photon_energies(g, n: int, median: float = 200.0, width: float = 1.3, top: float = 3500.0):
    """A broad (log-normal) spectrum of super-photon energies in m c^2, above
    the 2 m c^2 below which none is stored."""
    return torch.clamp(median * torch.exp(width * _normal(g, n)), 2.01, top)


def _decayed(g, tau, share: float):
    return torch.where(_unit(g, tau.numel()) < share, torch.full_like(tau, -1.0), tau)


def _beam(g, n: int, case: dict):
    """The collision's electrons, positrons and photons at step `start`."""
    sig = W.length(2e-6)
    dt = W.T_PERIOD / 100.0
    centre = (1000 - case["start"]) * dt

    def place(k):
        x, y, z = sig * _normal(g, 3, k)
        return {"x": x + centre, "y": y, "z": z, "w": torch.ones_like(x), "tau": _depths(g, k)}

    def move(s, u, spread):
        k = u.numel()
        ty, tz = spread * _normal(g, 2, k)
        norm = torch.sqrt(1.0 + ty * ty + tz * tz)
        s.update(ux=-u / norm, uy=u * ty / norm, uz=u * tz / norm)
        return s

    n_p, n_g = int(n * case["positrons"]), int(n * case["photons"])
    el = move(place(n), torch.clamp(4000.0 * (1.0 + 0.05 * _normal(g, n)), min=2.0), 0.01)
    po = move(place(n_p), _photon_energies(g, n_p, 500.0), 0.05)
    ph = move(place(n_g), _photon_energies(g, n_g), 0.05)
    ph["tau"] = _decayed(g, ph["tau"], case["dead"])
    return {"electron": el, "positron": po, "photon": ph}


def _foil(g, case: dict, w: dict):
    """The foil's electrons as the pulse finds them, with the positrons and
    photons of earlier steps among them."""
    src = {k: torch.as_tensor(v, device=DEV) for k, v in w["electrons"].items()}
    n = src["x"].numel()
    src["tau"] = _depths(g, n)
    # a tenth of the foil is already hot
    hot = _unit(g, n) < 0.1
    for k in ("ux", "uy", "uz"):
        src[k] = torch.where(hot, 60.0 * _normal(g, n), src[k])

    def among(k, scale):
        at = torch.randint(0, n, (k,), generator=g, device=DEV)
        d = _normal(g, 3, k)
        u = scale * d / d.norm(dim=0)
        return {"x": src["x"][at], "y": src["y"][at], "ux": u[0], "uy": u[1], "uz": u[2],
                "tau": _depths(g, k), "w": src["w"][at]}

    n_p, n_g = int(n * case["pairs"]), int(n * case["photons"])
    return {"electron": src, "positron": among(n_p, _photon_energies(g, n_p, 60.0)),
            "photon": among(n_g, _photon_energies(g, n_g, 30.0))}


# ---------------------------------------------------------------- states

_context = None


def _ctx():
    """One context a process, as a program keeps it."""
    global _context
    if _context is None:
        _context = Q.qp_init_tables(W.LAMBDA_M, 0)
    return _context


def _drop(ctx, handles):
    for h in handles:
        Q.qp_destroy_species(ctx, h)


class _State:
    pass


def _simulation(w: dict, particles: dict, case: dict, start: int, track: bool) -> _State:
    s = _State()
    s.case, s.start = case, start
    s.sim = sim = Simulation(w, precision=case["precision"], ctx=_ctx(), track_chi=track,
                             load=False)
    weakref.finalize(s, _drop, sim.ctx, [sp.handle for sp in sim.species.values()])
    s.rows, s.was = [], []
    for name in SPECIES:
        sp, arrays = sim.species[name], particles[name]
        n = arrays["x"].numel() if arrays else 0
        for nm, t in sp.t.items():
            if n:
                t[:n].copy_(arrays[nm])
                s.rows.append(t[:n])
        sp.n_live.fill_(n)
        Q.qp_reset_counters(sim.ctx, sp.handle)
    s.was = [t.clone() for t in s.rows]
    s.counts = sim.counts.clone()
    return s


def _put_back(s: _State):
    torch._foreach_copy_(s.rows, s.was)
    s.sim.counts.copy_(s.counts)
    s.sim.step_index = s.start


def _arrays(sim: Simulation) -> dict:
    out = {"counts": sim.counts}
    for name, sp in sim.species.items():
        if sp.cap:
            out[name] = sp.block
            if sp.nemit is not None:
                out[name + " events"] = sp.nemit
                out[name + " chi"] = sp.chi
    return out


def _read(d) -> dict:
    """One species' diagnostics: what the paper's figures show."""
    return {"whole": np.array([d.n_live, d.n_alive, d.n_emit, d.n_photon, d.n_photon_drop,
                               d.n_subthreshold, d.n_pair, d.n_pair_drop, d.n_saturated,
                               d.n_clamped, d.n_continuous, d.status], dtype=np.int64),
            "sums": np.array([d.weight, d.energy, d.px, d.py, d.pz, d.e_subthreshold,
                              d.e_dropped]),
            "chi": d.chi_mean, "spectrum": np.array(d.hist)}


def _plane_workload(case: dict) -> dict:
    n = case["n"]
    w = W.plane_wave_collision(n=n, n_steps=1000)
    n_g = int(n * case["photons"])
    w["capacity"] = {"electron": n, "positron": 0, "photon": n_g + n * (case["steps"] // 2 + 4)}
    return w


def _prepare_plane(case: dict, seed: int) -> _State:
    w = _plane_workload(case)
    w["params"]["seed"] = seed
    g = _gen(seed)
    n, n_g = case["n"], int(case["n"] * case["photons"])
    start = 40  # the electrons have met the wave's phases
    x = -2.0 * start * w["params"]["dt"] * _unit(g, n)
    zero = torch.zeros_like(x)
    el = {"x": x, "y": zero, "z": zero, "ux": -1999.0 * (1.0 + 0.02 * _normal(g, n)),
          "uy": 20.0 * _normal(g, n), "uz": zero, "tau": _depths(g, n),
          "w": torch.ones_like(x)}
    u = _photon_energies(g, n_g)
    zg = torch.zeros_like(u)
    ph = {"x": -5.0 * _unit(g, n_g), "y": zg, "z": zg, "ux": -u, "uy": 0.02 * u, "uz": zg,
          "tau": _depths(g, n_g), "w": torch.ones_like(u)}
    return _simulation(w, {"electron": el, "positron": None, "photon": ph}, case, start,
                       track=case["family"] == "plane")


def _prepare_foil(case: dict, seed: int) -> _State:
    family = case["family"]
    w = W.laser_on_foil(nx=case["nx"], ny=case["ny"], ppc=case["ppc"], seed=seed,
                        foil_cells=case["cells"], refill=case.get("fields") == "refill")
    w["params"]["seed"] = seed
    if family == "pic":
        # the solver's grid starts with the pulse at the foil
        w["field"]["pic"] = {"a0": 200.0, "w0": W.length(3 * W.LAMBDA_M),
                             "tau_fwhm": W.duration(30e-15),
                             "x_focus": (case["nx"] // 2) * w["field"]["dx"], "t_focus": 0.0,
                             "y_axis": 0.5 * case["ny"] * w["field"]["dy"]}
    p = _foil(_gen(seed), case, w)
    n, n_p, n_g = (p[k]["x"].numel() for k in SPECIES)
    more = n // 8 + 64
    w["capacity"] = {"electron": n + more, "positron": n_p + more,
                     "photon": n_g + n * (case["steps"] // 2 + 1)}
    s = _simulation(w, p, case, 250, track=False)
    s.grid = s.grid_was = None
    if family == "pic":
        s.grid, s.grid_was = s.sim._keep, [c.clone() for c in s.sim._keep]
    if family == "host":
        s.host, s.host_was, counts = {}, {}, {}
        for name in SPECIES:
            sp = s.sim.species[name]
            n = counts[name] = sp.count()
            s.host[name] = torch.zeros(sp.block.shape, dtype=torch.float64).pin_memory()
            s.host[name][:, :n].copy_(sp.block[:, :n])
            s.host_was[name] = s.host[name][:, :n].clone()
        s.states = s.sim.host_states(s.host, counts)
        s.host_counts = [counts[name] for name in SPECIES]
    return s


def _prepare_collision(case: dict, seed: int) -> _State:
    w = W.beam_collision(n=1, buffer=1)
    w["params"]["seed"] = seed
    n = case["n"]
    n_p, n_g = int(n * case["positrons"]), int(n * case["photons"])
    more = n // 4 + n_g // 8 + 256
    w["capacity"] = {"electron": n + more, "positron": n_p + more,
                     "photon": n_g + (n + n_p) * (case["steps"] // 3 + 1)}
    return _simulation(w, _beam(_gen(seed), n, case), case, case["start"], track=False)


def _prepare_cascade(case: dict, seed: int) -> _State:
    w = W.uniform_b_cascade(n=1)
    w["params"]["seed"] = seed
    g = _gen(seed)
    n = case["n"]
    n_p, n_g = int(n * case["positrons"]), int(n * case["photons"])

    def ring(k, u):
        phi, zero = 2.0 * math.pi * _unit(g, k), torch.zeros_like(u)
        return {"x": _normal(g, k), "y": _normal(g, k), "z": zero, "ux": u * torch.cos(phi),
                "uy": u * torch.sin(phi), "uz": zero, "tau": _depths(g, k),
                "w": torch.ones_like(u)}

    steps = case["steps"] * case["reads"]
    more = n // 2 + n_g // 4 + 64
    w["capacity"] = {"electron": n + more, "positron": n_p + more,
                     "photon": n_g + (n + n_p + more) * (steps // 4 + 1)}
    p = {"electron": ring(n, 3000.0 * (0.3 + 0.7 * _unit(g, n))),
         "positron": ring(n_p, _photon_energies(g, n_p, 300.0)),
         "photon": ring(n_g, _photon_energies(g, n_g))}
    return _simulation(w, p, case, 100, track=True)


def _prepare_coalesce(case: dict, seed: int) -> _State:
    n, sig = case["n"], W.length(2e-6)
    w = W.beam_collision(n=1, buffer=1)
    w["capacity"] = {"electron": 1, "positron": 1, "photon": n}
    g = _gen(seed)
    x, y, z = sig * _normal(g, 3, n)
    u = _photon_energies(g, n)
    ty, tz = 0.12 * _normal(g, 2, n)
    norm = torch.sqrt(1.0 + ty * ty + tz * tz)
    ph = {"x": x, "y": y, "z": z, "ux": -u / norm, "uy": u * ty / norm, "uz": u * tz / norm,
          "tau": _decayed(g, _depths(g, n), case["dead"]), "w": 0.5 + _unit(g, n)}
    none = {"electron": None, "positron": None, "photon": ph}
    s = _simulation(w, none, dict(case, precision="fp64"), 0, track=False)
    cells = (case["nx"], case["ny"], case["nz"])
    box = (-4.0 * sig, -4.0 * sig, -4.0 * sig) + tuple(8.0 * sig / c for c in cells)
    s.params = None
    if case["merge"]:
        s.params = Q.coalesce_params(box, cells, case["energy_bins"], case["direction_bins"],
                                     case["min_group"], seed=seed, step=30)
    s.box = box
    return s


def _close(engine, handles):
    torch.cuda.synchronize()
    engine.close()


def _prepare_serving(case: dict, seed: int) -> _State:
    rng = np.random.default_rng(seed)
    s = _State()
    s.requests, s.payloads = [], {}
    n_e = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]),
                             size=case["requests"])).astype(int)
    n_e[0] = case["n_max"]  # the stream's largest request is always among them
    for k in range(case["requests"]):
        r = {"id": k, "seed": int(seed) + k, "n": int(n_e[k]),
             "gamma": float(rng.uniform(1000.0, 5000.0)), "a0": float(rng.uniform(50.0, 500.0)),
             "n_steps": int(rng.integers(case["steps_min"], case["steps_max"] + 1)),
             "arrival_s": 0.0}
        w = W.beam_collision(n=r["n"], gamma=r["gamma"], a0=r["a0"], n_steps=r["n_steps"],
                             seed=r["seed"], buffer=8 * r["n"])
        s.requests.append(r)
        s.payloads[k] = w
    total = sum(8 * 26 * r["n"] * 8 + (1 << 20) for r in s.requests)
    s.engine = ServingEngine(max_slots=8, arena_bytes=int(1.1 * total), ctx=_ctx())
    weakref.finalize(s, _close, s.engine, None)
    return s


def prepare(case: dict, seed: int) -> _State:
    family = case["family"]
    make = {"plane": _prepare_plane, "fused": _prepare_plane, "foil": _prepare_foil,
            "host": _prepare_foil, "pic": _prepare_foil, "collision": _prepare_collision,
            "cascade": _prepare_cascade, "coalesce": _prepare_coalesce,
            "serving": _prepare_serving}[family]
    s = make(case, int(seed))
    s.case = case
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- a pass

def run(s: _State):
    case = s.case
    family = case["family"]
    if family == "serving":
        out = s.engine.run(s.requests, s.payloads)
        got = {}
        for r in out["results"]:
            for name in SPECIES:
                v = r[name]
                got["%d %s" % (r["id"], name)] = np.array([
                    v["n_live"], v["n_alive"], v["n_emit"], v["n_pair"], v["n_photon"],
                    v["n_dropped"], v["status"], r["work"]], dtype=np.int64)
                got["%d %s sums" % (r["id"], name)] = np.array([v["energy"], v["weight"]])
        return got
    if family == "host":
        for k, name in enumerate(SPECIES):
            n = s.host_counts[k]
            s.host[name][:, :n].copy_(s.host_was[name])
            s.states[k].count = n
        s.sim.step_index = s.start
        s.sim.run_host(s.states, case["steps"])
        return {"counts": np.array([s.states[k].count for k in range(3)], dtype=np.int64),
                **{name: s.host[name] for name in SPECIES}}
    _put_back(s)
    sim = s.sim
    if family == "coalesce":
        ph = sim.species["photon"]
        got = Q.qp_coalesce_photons(sim.ctx, ph.handle, s.params)
        return {"counts": np.array([got[k] for k in sorted(got)], dtype=np.int64), **ph.t}
    if family == "fused":
        sim.run_fused(case["steps"], case["steps"])
    elif family == "pic":
        torch._foreach_copy_(s.grid, s.grid_was)
        Q.qp_sort_species(sim.ctx, sim.species["electron"].handle, sim.field,
                          torch.cuda.current_stream().cuda_stream)
        sim.run(case["steps"])
        return {**_arrays(sim), "grid": s.grid}
    elif family == "cascade":
        reads = []
        for _ in range(case["reads"]):
            sim.run(case["steps"])
            reads.append([_read(sim.diagnostics(name)) for name in SPECIES])
        return {**_arrays(sim), "reads": reads}
    else:
        sim.run(case["steps"])
    return _arrays(sim)


# ---------------------------------------------------------------- bytes and operations

# FP operations of one particle-step that the physics cannot do without:
# gather or field model, push, quantum parameter, optical depth, motion
LEPTON_FLOPS, PHOTON_FLOPS = 250, 90


def _counts(case: dict):
    family = case["family"]
    if family in ("plane", "fused"):
        return case["n"], int(case["n"] * case["photons"])
    if family in ("foil", "host", "pic"):
        n = case["ny"] * case["cells"] * case["ppc"]
        return n + int(n * case["pairs"]), int(n * case["photons"])
    return (case["n"] + int(case["n"] * case["positrons"]),
            int(case["n"] * case["photons"]))


def work(case: dict) -> dict:
    """The state read once and written once a pass (a photon keeps its
    momentum), the grid and current once a cycle; particles made during the
    pass are left out."""
    family = case["family"]
    if family == "coalesce":
        # every photon read once, the survivors written
        return {"bytes": case["n"] * 8 * 8 * 1.3, "flops": case["n"] * 60}
    if family == "serving":
        lo, hi = case["n_min"], case["n_max"]
        mean_n = (hi - lo) / math.log(hi / lo) if hi > lo else hi
        n = hi + (case["requests"] - 1) * mean_n
        steps = 0.5 * (case["steps_min"] + case["steps_max"])
        return {"bytes": n * 2 * 8 * 8, "flops": n * steps * LEPTON_FLOPS}
    lep, pho = _counts(case)
    dims = 2 if family in ("foil", "host", "pic") else 3
    steps = case["steps"] * case.get("reads", 1)
    lep_b, pho_b = 2 * 8 * (dims + 4), 8 * (dims + 4) + 8 * (dims + 1)
    b = lep * lep_b + pho * pho_b
    if family in ("foil", "host", "pic"):
        # nodes under the particles (fixed fields), or the whole grid
        b += 6 * 4 * case["ny"] * case["cells"]
    if family == "pic":
        b += case["steps"] * case["ny"] * case["nx"] * (12 * 4 + 3 * 4)
    if case.get("fields") == "refill":
        b += case["steps"] * case["ny"] * case["nx"] * 2 * 4
    return {"bytes": b, "flops": steps * (lep * LEPTON_FLOPS + pho * PHOTON_FLOPS)}


# ---------------------------------------------------------------- 64-bit values

def exact(case: dict, seed: int):
    """Coalescence in 64-bit numpy.  The stepped cases have no such value:
    their events follow the library's own random streams and tables."""
    if case["family"] != "coalesce":
        return None
    s = _prepare_coalesce(case, int(seed))
    a = {nm: t.cpu().numpy().copy() for nm, t in s.sim.species["photon"].t.items()}
    n = case["n"]
    alive = a["tau"] >= 0.0
    u = np.stack([a["ux"], a["uy"], a["uz"]])
    en = np.sqrt((u * u).sum(axis=0))
    pairs, gone = [], ~alive
    if case["merge"]:
        x0, y0, z0, dx, dy, dz = s.box
        cells = [np.floor((a[k] - o) * (1.0 / d)) for k, o, d in
                 (("x", x0, dx), ("y", y0, dy), ("z", z0, dz))]
        ok = alive.copy()
        for c, m in zip(cells, (case["nx"], case["ny"], case["nz"])):
            ok &= (c >= 0) & (c < m)
        mant, ex = np.frexp(en)
        E, D = case["energy_bins"], case["direction_bins"]
        ebin = (ex + 1024).astype(np.int64) * E + np.floor((2.0 * mant - 1.0) * E).astype(np.int64)
        f = np.argmax(np.abs(u), axis=0)
        at = np.arange(n)
        dom = u[f, at]
        r = 1.0 / np.abs(dom)
        ia, ib = (np.minimum(np.floor((u[(f + q) % 3, at] * r + 1.0) * (0.5 * D)), D - 1)
                  .astype(np.int64) for q in (1, 2))
        cell = ((np.where(ok, cells[0], 0) * case["ny"] + np.where(ok, cells[1], 0)) * case["nz"]
                + np.where(ok, cells[2], 0)).astype(np.int64)
        key = ((cell * (4096 * E) + ebin) * 6 + 2 * f + (dom < 0.0)) * D * D + ia * D + ib
        who = at[ok][np.argsort(key[ok], kind="stable")]
        k = key[who]
        first = np.flatnonzero(np.r_[True, k[1:] != k[:-1]])
        size = np.diff(np.r_[first, len(k)])
        # groups above 256 merge in runs of 256
        cut = -(-size // 256)
        start = np.repeat(first, cut) + 256 * (np.arange(cut.sum())
                                               - np.repeat(np.cumsum(cut) - cut, cut))
        length = np.minimum(256, np.repeat(first + size, cut) - start)
        keep = length >= case["min_group"]
        start, length = start[keep], length[keep]
        members = who[np.repeat(start, length) + np.arange(length.sum())
                      - np.repeat(np.cumsum(length) - length, length)]
        edge = np.cumsum(length) - length

        def total(v):
            return np.add.reduceat(v[members], edge) if len(edge) else np.zeros(0)

        w_ = total(a["w"])
        e_ = total(a["w"] * en) / w_
        c = np.stack([total(a["w"] * q) / w_ for q in u])
        pos = np.stack([total(a["w"] * a[q]) / w_ for q in ("x", "y", "z")])
        lead = who[start]
        c2 = (c * c).sum(axis=0)
        dm = np.sqrt(np.maximum(e_ * e_ - c2, 0.0))
        ph = c / np.sqrt(c2)
        ref = u[:, lead]
        v = ref - (ref * ph).sum(axis=0) * ph
        v /= np.sqrt((v * v).sum(axis=0))
        pairs = [(lead[q], w_[q], pos[:, q], c[:, q] + dm[q] * v[:, q], c[:, q] - dm[q] * v[:, q])
                 for q in range(len(lead))]
        gone[members] = True
    # survivors in slot order, a merged pair in its first member's place
    takes = np.where(gone, 0, 1)
    if pairs:
        takes[np.array([p[0] for p in pairs])] = 2
    off = np.cumsum(takes) - takes
    out = {nm: v.copy() for nm, v in a.items()}
    kept = np.flatnonzero(~gone)
    for nm in ROWS3:
        out[nm][off[kept]] = a[nm][kept]
    if pairs:
        o = off[np.array([p[0] for p in pairs])]
        for sgn in (0, 1):
            for q, nm in enumerate(("x", "y", "z")):
                out[nm][o + sgn] = [p[2][q] for p in pairs]
            for q, nm in enumerate(("ux", "uy", "uz")):
                out[nm][o + sgn] = [p[3 + sgn][q] for p in pairs]
            out["w"][o + sgn] = [0.5 * p[1] for p in pairs]
    out["tau"] = None  # the merged photons draw fresh optical depths
    return {"counts": None, **out}
