"""Performance cases of the pairwise collision library.

Each case is the work of one call, or of one step's calls, as a simulation
code makes them through the binding (pcc.py, emission.py): binning, the
collision step with the commit of its secondaries, table builds, totals and
the differentiable expected-emission operator.

  listed()            the standing cases
  draw(rng)           one more case from the same ranges
  prepare(case, seed) what the caller holds before the call (inputs, context, tables)
  run(state)          one pass, returning its outputs whole
  work(case)          bytes and operations one pass cannot do without
  exact(case, seed)   the computed outputs in 64-bit torch, without the library
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1907_02814_gb300 import emission, pcc
from paper_1907_02814_gb300 import workloads as W

DEV = "cuda"
MEC2 = W.MEC2_MEV
CU = {"Z": 29, "Zstar": 5.0, "n_i": 8.5e28, "T_e": 100.0, "mass": W.MASS_CU}
AU = {"Z": 79, "n_i": 5.9e28, "T_e": 1000.0, "mass": W.MASS_AU}


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # 0D solid Cu, 64 cells of 64 electrons and 64 ions: one eager step of a
        # small run, where launches and host time are everything.
        {"name": "step_cu_64", "kind": "step", "plasma": "cu", "cells": 64, "law": "even", "mean": 64,
         "ions": 64.0, "photons": 0.0, "dt_fs": 0.1, "precision": "fp32", "graph_steps": 0},
        # 1D Au foil: 16384 cells, 31 ionization states, positions carried, the
        # foil run's time step; the time loop runs from a captured graph.
        {"name": "foil_au_graph", "kind": "step", "plasma": "au", "cells": 16384, "law": "poisson", "mean": 256,
         "ions": 64.0, "photons": 0.25, "dt_fs": 0.0074, "precision": "fp32", "graph_steps": 16},
        # 2^20 uneven solid-Cu cells (log-normal occupancy, ~2e8 electrons): one
        # eager step of the largest batched run.
        {"name": "step_cu_1m", "kind": "step", "plasma": "cu", "cells": 1 << 20, "law": "lognormal", "mean": 64,
         "ions": 0.147, "photons": 0.25, "dt_fs": 1.0, "precision": "fp32", "graph_steps": 0},
        # The FP64 path on the Au foil, as used to check a run against the
        # batched path.
        {"name": "foil_au_fp64", "kind": "step", "plasma": "au", "cells": 16384, "law": "poisson", "mean": 256,
         "ions": 64.0, "photons": 0.25, "dt_fs": 0.0074, "precision": "fp64", "graph_steps": 0},
        # A whole PIC step's calls on uneven cells: the moved electrons,
        # positrons and photons are binned again, collide, and their secondaries
        # are committed.
        {"name": "pic_cu_100k", "kind": "pic", "plasma": "cu", "cells": 100003, "law": "lognormal", "mean": 64,
         "ions": 0.147, "photons": 0.25, "dt_fs": 1.0},
        # First binning of a slab: few, very full cells, shuffled input with
        # positions (2048 cells of 8192 electrons).
        {"name": "bin_slab", "kind": "bin", "cells": 2048, "law": "even", "mean": 8192, "order": "shuffled", "x": True},
        # Binning of one small species, the photons of a thin slab early on.
        {"name": "bin_small", "kind": "bin", "cells": 60, "law": "poisson", "mean": 50, "order": "moved", "x": True},
        # Cross-section tables of the 31 ionization states of the foil, built
        # and read back (start-up, and again whenever the plasma state moves on).
        {"name": "tables_au_31", "kind": "tables", "materials": 31, "rows": 256, "cols": 256, "nodes": 8, "screening": 0},
        # Tables of one material with the numerically integrated screening.
        {"name": "tables_tfd", "kind": "tables", "materials": 1, "rows": 256, "cols": 256, "nodes": 8, "screening": 1},
        # Expected emission and its gradient over a full parameter set
        # (4096 plasma states x 512 samples, 64 nodes), one optimisation step.
        {"name": "emission_4096x512", "kind": "emission", "cells": 4096, "samples": 512, "nodes": 64, "spectrum": "loguniform"},
        # The same operator on a 1 MeV exponential electron source, two fifths
        # of it non-relativistic, odd sizes and a coarser rule.
        {"name": "emission_exp_333", "kind": "emission", "cells": 333, "samples": 77, "nodes": 48, "spectrum": "exponential"},
        # FP64 bookkeeping totals over the electrons of an uneven batch.
        {"name": "totals_256k", "kind": "totals", "cells": 262144, "law": "lognormal", "mean": 64, "photon": False},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "pic", "bin", "tables", "emission", "emission", "totals"])
    if kind in ("step", "pic"):
        plasma = rng.choice(["cu", "au"])
        law = rng.choice(["even", "poisson", "lognormal"])
        cells = _logint(rng, 64, 300000 if kind == "step" else 100000)
        mean = _logint(rng, 20, 400) if law != "lognormal" else _logint(rng, 16, 64)
        while cells * mean > 40_000_000:
            mean = max(16, mean // 2)
        case = {"kind": kind, "plasma": plasma, "cells": cells, "law": law, "mean": mean,
                "ions": float(_logint(rng, 8, 200)) if law != "lognormal" else round(rng.uniform(0.1, 1.0), 3),
                "photons": round(rng.choice([0.0, rng.uniform(0.05, 0.5)]), 3)}
        if kind == "pic":
            case["dt_fs"] = round(rng.uniform(0.1, 1.0), 3)
            return case
        case["dt_fs"] = round(math.exp(rng.uniform(math.log(0.0074), math.log(0.1))), 4)
        case["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        if case["precision"] == "fp64":
            case["cells"] = min(case["cells"], 16384)
        case["graph_steps"] = rng.choice([0, _logint(rng, 2, 32)])
        return case
    if kind == "bin":
        law = rng.choice(["even", "poisson", "lognormal"])
        cells = _logint(rng, 30, 200000)
        mean = _logint(rng, 10, 2000) if law != "lognormal" else _logint(rng, 8, 64)
        while cells * mean > 16_000_000:
            mean = max(8, mean // 2)
        return {"kind": "bin", "cells": cells, "law": law, "mean": mean, "order": rng.choice(["shuffled", "moved"]),
                "x": rng.random() < 0.5}
    if kind == "tables":
        tfd = 1 if rng.random() < 0.3 else 0
        return {"kind": "tables", "materials": 1 if tfd else _logint(rng, 1, 31), "rows": rng.randint(64, 256),
                "cols": rng.randint(64, 256), "nodes": rng.choice([4, 6, 8]), "screening": tfd}
    if kind == "emission":
        cells = _logint(rng, 8, 4096)
        return {"kind": "emission", "cells": cells, "samples": _logint(rng, 16, 512), "nodes": rng.randint(16, 64),
                "spectrum": rng.choice(["loguniform", "exponential"])}
    law = rng.choice(["even", "poisson", "lognormal"])
    return {"kind": "totals", "cells": _logint(rng, 64, 262144), "law": law, "mean": _logint(rng, 8, 64 if law == "lognormal" else 150),
            "photon": rng.random() < 0.4}


# ----------------------------------------------------------------- inputs --
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt * 7919) % (1 << 62))
    return g


def _counts(case, seed):
    """Electrons, ions, photons and positrons per cell (host arrays).  The
    occupancies belong to the case, their order over the cells to the seed, so
    that the totals and with them the buffer sizes are the case's own."""
    n = case["cells"]
    rng = np.random.default_rng([n, case["mean"], len(case["law"])])
    if case["law"] == "even":
        e = np.full(n, case["mean"], np.int64)
    elif case["law"] == "poisson":
        e = rng.poisson(case["mean"], n).astype(np.int64)
    else:
        e = W.lognormal_counts(rng, n, median=case["mean"])
    ions = case.get("ions", 0.0)
    i = W.ion_counts(rng, e, int(ions * e.sum())) if ions < 1.5 else np.full(n, int(ions), np.int64)
    g = rng.binomial(e, case.get("photons", 0.0))
    p = rng.binomial(e, 0.01)
    order = np.random.default_rng([int(seed), 11]).permutation(n)
    return e[order], i[order], g[order], p[order]


def _momenta(g, n, kind):
    u = torch.rand(n, device=DEV, generator=g, dtype=torch.float64)
    if kind == "photon":          # k ~ k^-2 on [2, 200] m_e c^2
        p = 1.0 / (0.5 - u * (0.5 - 1.0 / 200.0))
    else:
        if kind == "cu":          # exponential source, mean 1 MeV
            T = -torch.log1p(-u) / MEC2
        else:                     # E^-2 on 0.1 - 100 MeV
            a, b = 0.1 / MEC2, 100.0 / MEC2
            T = 1.0 / (1.0 / a - u * (1.0 / a - 1.0 / b))
        p = torch.sqrt(T * (T + 2.0))
    mu = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * 2.0 - 1.0
    phi = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * (2.0 * math.pi)
    s = torch.sqrt(1.0 - mu * mu)
    return (p * s * torch.cos(phi)).float(), (p * s * torch.sin(phi)).float(), (p * mu).float()


def _particles(case, seed, counts, kind, salt, with_x):
    """Device particle arrays of one species in cell and pid order.  kind:
    "cu" or "au" leptons, "photon", or "ion" (of case["plasma"])."""
    g = _gen(seed, salt)
    cnt = torch.as_tensor(counts, device=DEV)
    n = int(counts.sum())
    cell = torch.repeat_interleave(torch.arange(len(counts), device=DEV, dtype=torch.int32), cnt, output_size=n)
    if kind == "ion":
        m = CU if case["plasma"] == "cu" else AU
        sig = math.sqrt(m["T_e"] / (m["mass"] * MEC2 * 1e6))
        ux, uy, uz = (torch.randn(n, device=DEV, generator=g) * sig for _ in range(3))
        w = (m["n_i"] / cnt.clamp_min(1).float())[cell.long()]
    else:
        ux, uy, uz = _momenta(g, n, kind)
        if case.get("plasma", "cu") == "au":   # weights over three decades, mean density 3e25 m^-3
            wmean = 3e25 / case["mean"]
            w = wmean / (999.0 / (3.0 * math.log(10.0))) * 10.0 ** (3.0 * torch.rand(n, device=DEV, generator=g))
        else:
            w = torch.full((n,), CU["n_i"] / 64.0, device=DEV)
    x = (cell + torch.rand(n, device=DEV, generator=g)) * 2.4e-9 if with_x else None
    return {"ux": ux, "uy": uy, "uz": uz, "w": w, "pid": torch.arange(n, device=DEV), "cell": cell, "x": x, "n": n}


def _moved(parts, n_cells, seed, salt):
    """Particles after a push: half of them one cell to the left or right, in the storage order of before."""
    g = _gen(seed, salt)
    hop = torch.randint(0, 4, (parts["n"],), device=DEV, generator=g)
    step = (hop == 0).int() - (hop == 1).int()
    return dict(parts, cell=(parts["cell"] + step).clamp_(0, n_cells - 1))


def _shuffled(parts, seed, salt):
    perm = torch.randperm(parts["n"], device=DEV, generator=_gen(seed, salt))
    return {k: (v[perm] if torch.is_tensor(v) else v) for k, v in parts.items()}


NONE = {"n": 0, "ux": None, "uy": None, "uz": None, "w": None, "pid": None, "cell": None, "x": None}


def _room(n, cells, slack):
    return int(n + math.ceil(slack[1] * n) + (slack[0] + 1) * cells)


def _binned(ctx, parts, cells, slack, with_x):
    sp = pcc.DeviceSpecies.empty(cells, _room(parts["n"], cells, slack), device=DEV, with_x=with_x)
    pcc.bin(ctx, parts, cells, sp, slack_abs=slack[0], slack_rel=slack[1])
    return sp


def _plasma(case, seed):
    """(materials, material of each cell, ion mass, process mask)"""
    if case["plasma"] == "cu":
        mats = [pcc.material(CU["Z"], CU["Zstar"], CU["n_i"], CU["T_e"])]
        return mats, torch.zeros(case["cells"], dtype=torch.int32, device=DEV), CU["mass"], pcc.BREMS | pcc.TRIDENT | pcc.BH
    mats = [pcc.material(AU["Z"], float(z), AU["n_i"], AU["T_e"]) for z in range(10, 41)]
    mat = torch.randint(0, len(mats), (case["cells"],), device=DEV, generator=_gen(seed, 5), dtype=torch.int32)
    return mats, mat, AU["mass"], pcc.BREMS | pcc.BH


# region slack (absolute, relative): room for the secondaries of a long run
SLACK = {"em": (32, 0.1), "ep": (32, 0.1), "ph": (96, 2.0), "ion": (0, 0.0)}


def _emission_inputs(case, seed):
    rng = np.random.default_rng([int(seed), 23])
    n, m = case["cells"], case["samples"]
    params = np.stack([10.0 ** rng.uniform(25.0, 29.0, n), 10.0 ** rng.uniform(1.0, 4.0, n), rng.uniform(1.0, 28.0, n),
                       np.ones(n), np.ones(n)], 1)
    g = _gen(seed, 29)
    u = torch.rand((n, m), device=DEV, generator=g, dtype=torch.float64)
    if case["spectrum"] == "exponential":
        T = -torch.log1p(-u) / MEC2
    else:
        T = 0.5 * 400.0 ** u / MEC2
    w = torch.rand((n, m), device=DEV, generator=g) + 0.5
    gout = torch.randn((n, 3), device=DEV, generator=g)
    return torch.as_tensor(params, dtype=torch.float32, device=DEV), (1.0 + T).float(), w, gout


def _materials(case, seed):
    rng = np.random.default_rng([int(seed), 31])
    n = case["materials"]
    return [(79, float(z), 5.9e28, float(t)) for z, t in zip(rng.uniform(5.0, 60.0, n), 10.0 ** rng.uniform(1.5, 4.0, n))]


def prepare(case, seed):
    kind, cells = case["kind"], case.get("cells")
    s = {"case": case, "ctx": pcc.Context(0)}
    if kind in ("step", "pic"):
        mats, s["mat"], s["mass"], s["mask"] = _plasma(case, seed)
        s["ctx"].tables_build(mats, pcc.table_spec())
        s["dt"], s["seed"], s["step"] = case["dt_fs"] * 1e-15, int(seed) % (1 << 31) + 1, 0
        s["ledger"] = torch.zeros((cells, 4), device=DEV)
        e, i, g, p = _counts(case, seed)
        with_x = case["plasma"] == "au"
        ion = _particles(case, seed, i, "ion", 1, False)
        s["ion"] = _binned(s["ctx"], ion, cells, SLACK["ion"], False)
        em = _particles(case, seed, e, case["plasma"], 2, with_x)
        ph = _particles(case, seed, g, "photon", 3, with_x)
        if kind == "pic":
            ep = _particles(case, seed, p, case["plasma"], 4, with_x)
            s["in"] = {k: _moved(p, cells, seed, 40 + q) for q, (k, p) in enumerate((("em", em), ("ep", ep), ("ph", ph)))}
            for k, p in s["in"].items():
                s[k] = pcc.DeviceSpecies.empty(cells, _room(p["n"], cells, SLACK[k]), device=DEV, with_x=with_x)
            return s
        s["em"] = _binned(s["ctx"], em, cells, SLACK["em"], with_x)
        del em
        s["ph"] = _binned(s["ctx"], ph, cells, SLACK["ph"], with_x)
        del ph
        s["ep"] = _binned(s["ctx"], NONE, cells, SLACK["ep"], with_x)
        s["precision"] = pcc.FP64_PLAIN if case["precision"] == "fp64" else pcc.FP32_BATCHED
        if case["graph_steps"]:
            s["ctx"].steps_capture(cells, s["mat"], s["mass"], s["em"], s["ep"], s["ph"], s["ion"], s["dt"], s["seed"], 0,
                                   case["graph_steps"], mask=s["mask"], precision=s["precision"], ledger=s["ledger"])
    elif kind == "bin":
        e = _counts(case, seed)[0]
        p = _particles(case, seed, e, "photon" if case["order"] == "moved" else "cu", 2, case["x"])
        s["in"] = _moved(p, cells, seed, 41) if case["order"] == "moved" else _shuffled(p, seed, 41)
        s["out"] = pcc.DeviceSpecies.empty(cells, _room(p["n"], cells, (64, 0.25)), device=DEV, with_x=case["x"])
    elif kind == "tables":
        s["mats"] = [pcc.material(*m) for m in _materials(case, seed)]
        s["spec"] = pcc.table_spec(n_rows=case["rows"], n_cols=case["cols"], quad_nodes=case["nodes"], screening=case["screening"])
    elif kind == "emission":
        p, s["gamma"], s["w"], s["gout"] = _emission_inputs(case, seed)
        s["params"] = p.requires_grad_(True)
    else:
        e = _counts(case, seed)[0]
        s["sp"] = _binned(s["ctx"], _particles(case, seed, e, "photon" if case["photon"] else "cu", 2, False), cells, (8, 0.05), False)
    return s


# ------------------------------------------------------------------- pass --
def _species(sp):
    out = [sp.ux, sp.uy, sp.uz, sp.w, sp.pid, sp.cell_start, sp.cell_count]
    return out + [sp.x] if sp.x is not None else out


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind, cells = case["kind"], case.get("cells")
    if kind in ("step", "pic"):
        if kind == "pic":
            for k in ("em", "ep", "ph"):
                pcc.bin(ctx, s["in"][k], cells, s[k], slack_abs=SLACK[k][0], slack_rel=SLACK[k][1])
        if case.get("graph_steps"):
            ctx.steps_launch()
        else:
            pcc.collide(ctx, cells, s["mat"], s["mass"], s["em"], s["ep"], s["ph"], s["ion"], s["dt"], s["seed"], s["step"],
                        mask=s["mask"], precision=s.get("precision", pcc.FP32_BATCHED), ledger=s["ledger"])
            for k in ("em", "ep", "ph"):
                pcc.append_secondaries(ctx, cells, s[k])
            s["step"] += 1
        return {"em": _species(s["em"]), "ep": _species(s["ep"]), "ph": _species(s["ph"]), "ledger": s["ledger"]}
    if kind == "bin":
        pcc.bin(ctx, s["in"], cells, s["out"], slack_abs=64, slack_rel=0.25)
        return _species(s["out"])
    if kind == "tables":
        ctx.tables_build(s["mats"], s["spec"])
        return ctx.tables_read()
    if kind == "emission":
        out = emission.expected_emission(ctx, 29, s["params"], s["gamma"], s["w"], n_quad=case["nodes"])
        grad, = torch.autograd.grad(out, s["params"], s["gout"])
        return [*out.detach().unbind(1), *grad.unbind(1)]
    return pcc.totals(ctx, cells, s["sp"], is_photon=case["photon"])


def work(case):
    """A particle record is u, w (16 B) and id (8 B), with x 28 B; a cell has a start and a count per species."""
    kind, n = case["kind"], case.get("cells", 0)
    mean = case.get("mean", 0)
    e = n * (mean * (3.0 if case.get("law") == "lognormal" else 1.0))
    if kind in ("step", "pic"):
        # the weights of every particle and ion (the pair coefficient needs
        # their sums), the cell arrays, and the accept uniforms of every pair:
        # ten rounds of two wide products for a draw of four e- or eight photon pairs
        ions = case["ions"] * e if case["ions"] < 1.5 else case["ions"] * n
        ph = case["photons"] * e
        pairs = max(e, ions) / 4 + (max(ph, ions) / 8 if ph else 0)
        steps = max(case.get("graph_steps", 0), 1)
        b = 4.0 * (e + ions + ph) + 52.0 * n
        if kind == "pic":
            rec = 28.0 if case["plasma"] == "au" else 24.0
            b += (2 * rec + 4.0) * (1.01 * e + ph) + 36.0 * n
        return {"bytes": steps * b, "flops": steps * 60.0 * pairs}
    if kind == "bin":
        rec = 28.0 if case["x"] else 24.0
        return {"bytes": e * (2 * rec + 4.0) + 12.0 * n, "flops": 0.0}
    if kind == "tables":
        cells = case["rows"] * case["cols"]
        evals = case["materials"] * cells * case["nodes"] * 2.0 + 2.0 * cells * case["nodes"]
        return {"bytes": 8.0 * cells * (2 * case["materials"] + 2) * 2.0, "flops": evals * (12.0 * 10 * 40 if case["screening"] else 120.0)}
    if kind == "emission":
        nodes = float(n) * case["samples"] * case["nodes"]
        return {"bytes": 16.0 * n * case["samples"] + 100.0 * n, "flops": 180.0 * nodes}
    return {"bytes": 16.0 * e + 8.0 * n, "flops": 16.0 * e}


# ------------------------------------------------------- 64-bit references --
ALPHA, R_E, R_C, C_LIGHT = 7.2973525693e-3, 2.8179403262e-15, 3.8615926796e-13, 299792458.0
EPS0, Q_E = 8.8541878128e-12, 1.602176634e-19


def _f_c(Z):
    """Coulomb correction with four terms of its series."""
    a2 = (ALPHA * Z) ** 2
    n = np.arange(2, 200001, dtype=np.float64)
    tail = [math.fsum(n[::-1] ** -s) + 200000.5 ** (1 - s) / (s - 1) for s in (3.0, 5.0, 7.0, 9.0)]
    return a2 * (1.0 / (1.0 + a2) + sum((-a2) ** k * t for k, t in enumerate(tail)))


def _screening(Z, n_i, T_e, zs, s_tf, s_d):
    """L_TF, L_D, eta_D, I_TFD and the reduced length (torch, 64 bits)."""
    ltf = s_tf * Z ** (-1.0 / 3.0) / ALPHA
    ri = (3.0 / (4.0 * math.pi * n_i)) ** (1.0 / 3.0)
    lam = torch.sqrt(EPS0 * T_e / (Q_E * n_i * zs * (zs + 1.0)))
    ld = s_d * torch.maximum(lam, ri) / R_C
    ed = zs / Z
    et = 1.0 - ed
    a, b = ltf ** 2, ld ** 2
    h = lambda v: torch.log1p(v) - v / (1.0 + v)
    i_tfd = 0.5 * et ** 2 * h(a) + 0.5 * ed ** 2 * h(b) + et * ed * (b * torch.log1p(a) - a * torch.log1p(b)) / (b - a)
    # h(L^2) = 2 I_TFD: Newton in v = ln(1 + L^2), the last step differentiable
    with torch.no_grad():
        v = 2.0 * i_tfd + 1.0
        for _ in range(60):
            v = v - (v + torch.exp(-v) - 1.0 - 2.0 * i_tfd) / (1.0 - torch.exp(-v))
    v = v - (v + torch.exp(-v) - 1.0 - 2.0 * i_tfd) / (1.0 - torch.exp(-v))
    return ltf, ld, ed, i_tfd, torch.sqrt(torch.expm1(v))


def _yukawa(L, d, omd):
    """I1 and I2 of the reduced potential at delta = d = 1 - omd."""
    u, l2 = L * d, L * L
    u2 = u * u
    rho = l2 / (1.0 + l2)
    A = torch.atan(L * omd / (1.0 + L * u))
    lnr = torch.log1p(l2 * omd * (1.0 + d) / (1.0 + u2))
    i1 = -u * A - 0.5 * rho * omd ** 2 + 0.5 * lnr
    i2 = -2.0 * u2 * u * A + 0.5 * (1.0 + 3.0 * u2) * lnr + 3.0 * rho * u2 * torch.log(d) - 0.5 * rho * omd * (1.0 + d - 4.0 * u2)
    return i1, i2


def _rel_shape(g, k, gk, i1, i2, fc):
    eps = gk / g
    return (1.0 + eps ** 2) * (i1 + 1.0 - fc) - (2.0 / 3.0) * eps * (i2 + 5.0 / 6.0 - fc)


def _nr_shape(Z, T1, T2, k, ltf, ld, ed):
    """Non-relativistic bracket with the Elwert factor, over 4 Z^2 r_e^2 alpha / k."""
    p1, p2 = torch.sqrt(T1 * (T1 + 2.0)), torch.sqrt(T2 * (T2 + 2.0))
    qm = k * (T1 + T2 + 2.0) / (p1 + p2)
    P = 4.0 * p1 * p2
    et = 1.0 - ed
    a, b = ltf ** 2, ld ** 2
    da, db = 1.0 + qm ** 2 * a, 1.0 + qm ** 2 * b
    ra, rb = P * a / da, P * b / db
    la, lb = torch.log1p(ra), torch.log1p(rb)
    br = 0.5 * et ** 2 * (la - ra / (da + P * a)) + 0.5 * ed ** 2 * (lb - rb / (db + P * b)) + et * ed / (b - a) * (b * la - a * lb)
    b1, b2 = p1 / (1.0 + T1), p2 / (1.0 + T2)
    az = 2.0 * math.pi * Z * ALPHA
    return 4.0 / (3.0 * p1 ** 2) * br * (b1 / b2) * torch.expm1(-az / b1) / torch.expm1(-az / b2)


def _exact_emission(case, seed):
    p32, gamma32, w32, gout = _emission_inputs(case, seed)
    Z, n, m = 29, case["cells"], case["samples"]
    gx, gw = np.polynomial.legendre.leggauss(case["nodes"])
    half = -0.5 * math.log(1e-7)
    l = torch.as_tensor(half * (gx - 1.0), device=DEV)
    hw = torch.as_tensor(half * gw, device=DEV)
    x, omx = torch.exp(l), -torch.expm1(l)
    outs, grads = [], []
    chunk = max(1, 12_000_000 // (m * case["nodes"]))
    fc_val = _f_c(Z)
    for c0 in range(0, n, chunk):
        par = p32[c0:c0 + chunk].double().requires_grad_(True)
        gamma, w = gamma32[c0:c0 + chunk].double(), w32[c0:c0 + chunk].double()
        n_i, T_e, zs, s_tf, s_d = par.unbind(1)
        ltf, ld, ed, _, lr = _screening(Z, n_i, T_e, zs, s_tf, s_d)
        cell = torch.arange(gamma.shape[0], device=DEV)[:, None].expand_as(gamma)
        R = torch.zeros_like(n_i)
        P = torch.zeros_like(n_i)
        for rel in (False, True):
            sel = (gamma > 2.0) if rel else (gamma <= 2.0) & (gamma > 1.0)
            ci, g = cell[sel], gamma[sel][:, None]
            if g.numel() == 0:
                continue
            T = g - 1.0
            k, T2 = T * x, T * omx
            if rel:
                gk = 1.0 + T2
                d = k / (2.0 * g * gk)
                i1, i2 = _yukawa(lr[ci][:, None], d, 1.0 - d)
                f = _rel_shape(g, k, gk, i1, i2, torch.where(g > 100.0, fc_val, 0.0))
            else:
                f = _nr_shape(Z, T, T2, k, ltf[ci][:, None], ld[ci][:, None], ed[ci][:, None])
            f = f.clamp_min(0.0)
            wb = w[sel] * torch.sqrt(T * (T + 2.0))[:, 0] / g[:, 0]
            R = R.index_add(0, ci, wb * (f * hw).sum(1))
            P = P.index_add(0, ci, wb * (f * k * hw).sum(1))
        lt = torch.log((gamma + 4.5) / 6.89)
        sig_t = torch.where(gamma >= 3.0, 5.22e-34 * Z * Z * lt ** 3, 0.0)
        pair = (w * torch.sqrt(gamma ** 2 - 1.0) / gamma * sig_t).sum(1)
        c0_ = 4.0 * Z * Z * R_E ** 2 * ALPHA * C_LIGHT
        out = torch.stack([n_i * c0_ * R, n_i * C_LIGHT * pair, n_i * c0_ * P], 1)
        grad, = torch.autograd.grad(out, par, gout[c0:c0 + chunk].double())
        outs.append(out.detach())
        grads.append(grad)
    return [*torch.cat(outs).unbind(1), *torch.cat(grads).unbind(1)]


def _panels(cols, log, ly):
    """Panel edges and their column: one per column interval, graded ones at the ends."""
    t = torch.arange(cols, device=DEV, dtype=torch.float64) / (cols - 1)
    e = ly * (1.0 - t) if log else t
    a, b, col = [e[:-1]], [e[1:]], [torch.arange(cols - 1, device=DEV)]
    grade = 0.25 ** torch.arange(1, 13, device=DEV, dtype=torch.float64)
    for left in ([False] if log else [False, True]):
        c = 0 if left else cols - 2
        lo, hi = e[c], e[c + 1]
        cut = torch.cat([hi[None], lo + (hi - lo) * grade, lo[None]]) if left else torch.cat([lo[None], hi - (hi - lo) * grade, hi[None]])
        a.append(torch.minimum(cut[:-1], cut[1:]))
        b.append(torch.maximum(cut[:-1], cut[1:]))
        col.append(torch.full((13,), c, device=DEV))
        b[0] = b[0].clone()
        b[0][c] = a[0][c]      # the plain panel of a graded column is empty
    return torch.cat(a), torch.cat(b), torch.cat(col)


def _tfd_i12(ltf, ld, ed, d):
    """I1 and I2 of the full potential: 12-point Gauss-Legendre on unit panels of t = ln u from 0 down to ln d."""
    gx, gw = np.polynomial.legendre.leggauss(12)
    t0 = torch.log(d)
    i1, i2 = torch.zeros_like(d), torch.zeros_like(d)
    hi = 0.0
    low = float(t0.min())
    while hi > low:
        lo = torch.clamp_min(t0, hi - 1.0)
        h, mid = 0.5 * (hi - lo).clamp_min(0.0), 0.5 * (hi + lo)
        for xq, wq in zip(gx, gw):
            t = mid + h * xq
            u2, lr = torch.exp(2.0 * t), t - t0
            ir = torch.exp(-lr)
            f2 = ((1.0 - ed) * ltf ** 2 * u2 / (1.0 + ltf ** 2 * u2) + ed * ld ** 2 * u2 / (1.0 + ld ** 2 * u2)) ** 2
            i1 += h * wq * torch.expm1(-lr) ** 2 * f2
            i2 += h * wq * (1.0 + (3.0 - 6.0 * lr) * ir ** 2 - 4.0 * ir ** 3) * f2
        hi -= 1.0
    return i1, i2


def _row_table(shape, rows, cols, nodes, log, ly):
    a, b, col = _panels(cols, log, ly)
    gx, gw = (torch.as_tensor(v, device=DEV) for v in np.polynomial.legendre.leggauss(nodes))
    h, mid = 0.5 * (b - a), 0.5 * (a + b)
    v = mid[:, None] + h[:, None] * gx
    out = []
    for r0 in range(0, rows.numel(), 64):
        f = shape(rows[r0:r0 + 64][:, None, None], v[None])
        part = (f * gw).sum(2) * h
        out.append(torch.zeros((part.shape[0], cols - 1), device=DEV, dtype=torch.float64).index_add(1, col, part))
    cum = torch.cumsum(torch.cat(out), 1)
    tot = cum[:, -1]
    cdf = torch.cat([torch.zeros_like(tot)[:, None], cum / tot[:, None]], 1)
    return tot, torch.where((tot > 0.0)[:, None], cdf, torch.linspace(0.0, 1.0, cols, device=DEV, dtype=torch.float64))


def _exact_tables(case, seed):
    R, C, Q, tfd = case["rows"], case["cols"], case["nodes"], case["screening"]
    t_min, t_max = 0.002, 1999.0
    rows = t_min * (t_max / t_min) ** (torch.arange(R, device=DEV, dtype=torch.float64) / (R - 1))
    tab = {k: [] for k in ("brems_sigma", "brems_cdf", "bh_sigma", "bh_cdf", "screening")}
    for Z, zs, n_i, T_e in _materials(case, seed):
        t = lambda v: torch.tensor(float(v), device=DEV, dtype=torch.float64)
        ltf, ld, ed, i_tfd, lr = _screening(Z, t(n_i), t(T_e), t(zs), t(1.0), t(1.0))
        fcv = _f_c(Z)
        unit = 4.0 * Z * Z * R_E ** 2 * ALPHA

        def screen_i12(d, omd):
            return _tfd_i12(ltf, ld, ed, d) if tfd else _yukawa(lr, d, omd)

        def brems(T, v):
            x, omx = torch.exp(v), -torch.expm1(v)
            if float(T.max()) > 1.0 >= float(T.min()):      # both regimes in these rows: row by row
                return torch.cat([brems(T[i:i + 1], v) for i in range(T.shape[0])])
            k, g = T * x, 1.0 + T
            if float(T.max()) <= 1.0:
                f = _nr_shape(Z, T, T * omx, k, ltf, ld, ed)
            else:
                gk = 1.0 + T * omx
                d = k / (2.0 * g * gk)
                f = _rel_shape(g, k, gk, *screen_i12(d, 1.0 - d), torch.where(g > 100.0, fcv, 0.0)).clamp_min(0.0)
            return unit * f            # dsigma/dk k per d ln k

        def bethe_heitler(T, y):
            k, gp = 2.0 + T, 1.0 + y * T
            gm = k - gp
            d = k / (2.0 * gp * gm)
            i1, i2 = screen_i12(d.clamp_max(1.0), (1.0 - d).clamp_min(0.0))
            f = ((gp ** 2 + gm ** 2) * (i1 + 1.0) + (2.0 / 3.0) * gp * gm * (i2 + 5.0 / 6.0)) / k ** 3
            return unit * f.clamp_min(0.0) * T

        for name, shape, log in (("brems", brems, True), ("bh", bethe_heitler, False)):
            sig, cdf = _row_table(shape, rows, C, Q, log, -7.0 * math.log(10.0))
            tab[name + "_sigma"].append(sig)
            tab[name + "_cdf"].append(cdf)
        tab["screening"].append(torch.stack([ltf, ld, 1.0 - ed, ed, i_tfd, lr, t(fcv), t(Z)]))

    def pair(T, v):
        g, y = 3.0 + T, torch.exp(v)
        gp = 2.0 + y * T
        pre = (R_E * ALPHA) ** 2
        x2 = 1.0 / g ** 2
        q, L = x2 / (1.0 - x2), -torch.log(x2)
        c = 4.0 * q * L - (4.0 / 3.0) * x2 + x2 ** 2 / 6.0
        cz = 3.0 * q * (1.0 - q * L) - 2.6 * x2 + 1.75 * x2 ** 2 - 0.9 * x2 ** 3 + 0.2 * x2 ** 4
        cr = -1.5 * q * (1.0 - q * L) + 0.8 * x2 - 0.125 * x2 ** 2 - 0.05 * x2 ** 3 + 0.025 * x2 ** 4
        nr = pre / 32.0 * (2.0 * torch.log(g) - 161.0 / 60.0 + c + cr + cz) * (y * T) ** 3
        r = 56.0 / (9.0 * math.pi) * pre * torch.log(gp) * torch.log(g / gp) / gp
        return torch.where((nr > 0.0) & (r > 0.0), nr * r / (nr + r), 0.0) * T * y

    def split(T, y):
        gp = 2.0 + T
        a = 1.0 + y * T
        b = gp - a
        return ((a ** 2 + b ** 2 + (2.0 / 3.0) * a * b) * torch.log(a * b / gp)).clamp_min(0.0) * T

    out = {k: torch.stack(v) for k, v in tab.items()}
    out["tri_gp_cdf"] = _row_table(pair, rows, C, Q, True, math.log(1e-5))[1]
    out["tri_split_cdf"] = _row_table(split, rows, C, Q, False, 0.0)[1]
    return out


def _exact_bin(case, seed):
    """The arrays as binning lays them out: cell regions with slack, ids ascending within a cell."""
    s = prepare(case, seed)
    p, n_cells = s["in"], case["cells"]
    order = torch.argsort(p["pid"])
    order = order[torch.argsort(p["cell"][order], stable=True)]
    cell = p["cell"][order].long()
    cnt = torch.bincount(cell, minlength=n_cells)
    room = cnt + torch.clamp_min(torch.ceil(0.25 * cnt.double()).long(), 64)
    start = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(room, 0)])
    first = torch.cumsum(cnt, 0) - cnt
    slot = start[cell] + torch.arange(p["n"], device=DEV) - first[cell]

    def put(v):
        out = torch.zeros(s["out"].capacity, dtype=torch.float64, device=DEV)
        out[slot] = v[order].double()
        return out

    f = [put(p[k]) for k in ("ux", "uy", "uz", "w")] + [None, None, None]
    return f + [put(p["x"])] if case["x"] else f


def exact(case, seed):
    """Collision steps draw discrete events from the library's own random
    streams, so they have no closed 64-bit value."""
    kind = case["kind"]
    if kind == "emission":
        return _exact_emission(case, seed)
    if kind == "tables":
        return _exact_tables(case, seed)
    if kind == "bin":
        return _exact_bin(case, seed)
    if kind == "totals":
        e = _counts(case, seed)[0]
        p = _particles(case, seed, e, "photon" if case["photon"] else "cu", 2, False)
        u = torch.sqrt(p["ux"].double() ** 2 + p["uy"].double() ** 2 + p["uz"].double() ** 2)
        w = p["w"].double()
        return torch.stack([w.sum(), (w * (u if case["photon"] else torch.sqrt(1.0 + u * u))).sum(), (w * u).sum()])
    return None
