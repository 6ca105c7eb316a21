"""Timed cases: what a user of the library has it do, through its public entry points.

Two kinds of work.  Engine runs (`nefe.Context`): a block of MD steps of one or many systems, then
what a switching run is made for (W, the Hamiltonian's terms, pressure, box) and the state.  Calls
on the caller's own tensors and trajectories: neighbour list and forces, the differentiable energy
(`autograd.sw_energy`), the checkpointed adjoint of the switching work (`nefe.Adjoint`).

Outputs of the FP32 kernels come back in FP64 arrays; they are handed on as float32, which is what
they carry.  Outputs of the FP64 kernels stay float64; cell and list entries stay whole numbers.
"""
import math

import numpy as np
import torch

from paper_2103_10449_gb300 import autograd as AG
from paper_2103_10449_gb300 import inputs as I
from paper_2103_10449_gb300 import nefe as N

KB = 8.617333262e-5                                  # eV/K
MVV2E = 1.66053906660e-23 / 1.602176634e-19          # (g/mol) A^2/ps^2 -> eV
MASS = 28.0855
UF = (25.0, 2.0, 2200.0, 8.0)                        # the liquid's reference fluid: p, sigma, T, rc
GPA = 160.21766340                                   # eV/A^3 -> GPa


# ------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one small crystal, FP64, 400 K: a convergence check of a switching protocol at the desk;
        # every step is launches and latency
        {"name": "fl_64_fp64", "kind": "fl", "reps": 1, "cells": "2x2x2", "vac": 0, "fp64": True, "skin": 0.5,
         "T": 400.0, "tune": False, "steps": 256},
        # the README's example: one 8000-atom crystal with the defaults
        {"name": "fl_8000_fp32", "kind": "fl", "reps": 1, "cells": "10x10x10", "vac": 0, "fp64": False, "skin": 0.5,
         "T": 1000.0, "tune": False, "steps": 320},
        # the FP64 arm of the free-energy error estimate: 16 realisations of 8000 atoms
        {"name": "fl_8000x16_fp64", "kind": "fl", "reps": 16, "cells": "10x10x10", "vac": 0, "fp64": True, "skin": 0.5,
         "T": 1000.0, "tune": False, "steps": 32},
        # the benchmark's batch: 128 realisations of 8000 atoms, autotuned, skin 1.6 A
        {"name": "fl_8000x128_fp32", "kind": "fl", "reps": 128, "cells": "10x10x10", "vac": 0, "fp64": False,
         "skin": 1.6, "T": 1000.0, "tune": True, "steps": 320},
        # coexistence integration of 64 diamond / beta-tin pairs of uneven sizes, autotuned
        {"name": "dcci_64pairs_fp32", "kind": "dcci", "pairs": 64, "lo": 512, "hi": 32768, "skin": 0.7, "tune": True,
         "steps": 160},
        # reversible scaling at constant pressure, 4 realisations of each phase, as the phase
        # diagram's runs are set up (barostats on, defaults)
        {"name": "rs_npt_12x8000_fp32", "kind": "rs", "reps": 4, "atoms": 8000, "P": 10.0, "skin": 0.7, "steps": 160},
        # switching the liquid to its reference fluid, 4 realisations
        {"name": "uf_switch_4x8000_fp32", "kind": "uf", "reps": 4, "atoms": 8000, "skin": 0.7, "steps": 64},
        # a host program that hands in all positions and velocities, runs one block and reads the
        # results, block after block
        {"name": "host_io_32x8000_fp32", "kind": "io", "reps": 32, "cells": "10x10x10", "skin": 0.7, "T": 1000.0,
         "steps": 32},
        # list and forces of a small crystal with vacancies (a static relaxation's inner call)
        {"name": "forces_1723_fp64", "kind": "forces", "form": "crystal", "cells": "6x6x6", "vac": 5, "fp64": True,
         "skin": 0.5},
        # list and forces of a million-atom crystal
        {"name": "forces_1000000_fp32", "kind": "forces", "form": "crystal", "cells": "50x50x50", "vac": 0,
         "fp64": False, "skin": 0.5},
        # the differentiable energy, forward and backward, on the liquid of the fitting workload
        {"name": "grad_liquid_32768_fp64", "kind": "grad", "form": "liquid", "atoms": 32768, "fp64": True, "skin": 0.5},
        # the switching work of that liquid and its gradient: forward run and reverse sweep
        {"name": "adjoint_liquid_32768", "kind": "adjoint", "sched": "rs", "atoms": 32768, "steps": 24, "every": 8},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_cells(rng, lo, hi):
    """Cell counts of a crystal of about lo .. hi atoms (log-uniform), the axes of uneven lengths."""
    m = max(8.0, _logint(rng, lo, hi) / 8.0)
    a, b = rng.uniform(0.7, 1.4), rng.uniform(0.7, 1.4)
    g = m ** (1.0 / 3.0)
    return [max(2, int(round(g * a))), max(2, int(round(g * b))), max(2, int(round(g / (a * b))))]


def draw(rng):
    kind = rng.choice(["fl", "fl", "fl", "dcci", "rs", "uf", "io", "forces", "forces", "grad", "grad", "adjoint"])
    name = lambda c: "x".join(str(v) for v in c)  # noqa: E731
    if kind == "fl":
        fp64 = rng.random() < 0.35
        c = _draw_cells(rng, 64, 12000)
        n = 8 * c[0] * c[1] * c[2]
        reps = min(_logint(rng, 1, 64), max(1, (100000 if fp64 else 600000) // n))
        steps = rng.choice([32, 50, 96]) if fp64 else rng.choice([64, 75, 160, 256])
        # the wide skin is the crystal batch's setting; it needs a box of two cells per axis
        skin = rng.choice([0.5, 0.7, 1.0] if fp64 else [0.5, 0.7, 1.0, 1.6])
        return {"kind": kind, "reps": reps, "cells": name(c), "vac": rng.choice([0, 0, 1, 3]), "fp64": fp64, "skin": skin,
                "T": rng.choice([400.0, 700.0, 1000.0]), "tune": rng.random() < 0.4, "steps": steps}
    if kind == "dcci":
        return {"kind": kind, "pairs": _logint(rng, 1, 32), "lo": 512, "hi": _logint(rng, 1024, 20000), "skin": 0.7,
                "tune": rng.random() < 0.5, "steps": rng.choice([64, 100, 128])}
    if kind == "rs":
        return {"kind": kind, "reps": _logint(rng, 1, 6), "atoms": _logint(rng, 700, 12000),
                "P": rng.choice([0.0, 5.0, 10.0]), "skin": 0.7, "steps": rng.choice([64, 100, 160])}
    if kind == "uf":
        return {"kind": kind, "reps": _logint(rng, 1, 4), "atoms": _logint(rng, 2500, 9000), "skin": rng.choice([0.5, 0.7]),
                "steps": rng.choice([32, 45, 64])}
    if kind == "io":
        c = _draw_cells(rng, 500, 12000)
        return {"kind": kind, "reps": min(_logint(rng, 1, 32), max(1, 256000 // (8 * c[0] * c[1] * c[2]))),
                "cells": name(c), "skin": rng.choice([0.5, 0.7]), "T": 1000.0, "steps": rng.choice([32, 48])}
    if kind in ("forces", "grad"):
        c = {"kind": kind, "form": rng.choice(["crystal", "crystal", "liquid"]), "fp64": rng.random() < 0.5,
             "skin": rng.choice([0.3, 0.5, 0.7])}
        top = 300000 if kind == "forces" else 120000
        if c["form"] == "crystal":
            c["cells"], c["vac"] = name(_draw_cells(rng, 64, top)), rng.choice([0, 1, 7])
        else:
            c["atoms"] = _logint(rng, 700, top)
        return c
    return {"kind": "adjoint", "sched": rng.choice(["rs", "fl"]), "atoms": _logint(rng, 700, 16000),
            "steps": rng.choice([9, 16, 24]), "every": rng.choice([4, 8, 45])}


# --------------------------------------------------------------------------------------- inputs
def _cells(case):
    return [int(v) for v in case["cells"].split("x")]


def _crystal(nx, ny, nz, T, seed, vac=0):
    """Ideal sites, thermal positions (independent harmonic displacements at T, k = 6.1 eV/A^2 as
    the crystal's Einstein constant) and velocities of a diamond crystal with vac vacancies."""
    r0, box = I.diamond(nx, ny, nz)
    rng = np.random.default_rng(seed)
    if vac:
        r0 = np.delete(r0, rng.choice(len(r0), size=vac, replace=False), axis=0)
    x = r0 + rng.standard_normal(r0.shape) * math.sqrt(KB * T / 6.1)
    return r0, x, _velocities(len(r0), T, seed), box


def _velocities(n, T, seed):
    return I.gaussian_velocities(n, math.sqrt(KB * T / (MASS * MVV2E)), seed)


def _liquid(n, seed, density=0.05425):
    """Disordered positions at the liquid's density: a cubic grid (2.64 A) with as many sites as
    needed, n of them taken, each displaced by up to 0.35 A per axis (no pair below 1.9 A)."""
    L = (n / density) ** (1.0 / 3.0)
    m = int(math.ceil(n ** (1.0 / 3.0) - 1e-9))
    while m ** 3 < n:
        m += 1
    rng = np.random.default_rng(seed)
    k = rng.permutation(m ** 3)[:n]
    g = np.stack([k // (m * m), (k // m) % m, k % m], axis=1)
    h = L / m
    amp = min(0.35, 0.5 * (h - 1.9))
    x = (g + 0.5) * h + rng.uniform(-amp, amp, (n, 3))
    return x, np.array([L, L, L])


def _seed(seed, k):
    return (int(seed) * 1000003 + 7919 * k) % (1 << 31)


def _atoms(case):
    """Atoms of one pass, summed over its systems."""
    k = case["kind"]
    if k in ("fl", "io"):
        c = _cells(case)
        return case["reps"] * (8 * c[0] * c[1] * c[2] - case.get("vac", 0))
    if k == "dcci":
        total = 0
        for n in I.log_uniform_sizes(case["pairs"], case["lo"], case["hi"], seed=2021):
            a, b = I.diamond_cells_for(n), I.beta_tin_cells_for(n)
            total += 8 * a[0] * a[1] * a[2] + 4 * b[0] * b[1] * b[2]
        return total
    if k == "rs":
        return 3 * case["reps"] * case["atoms"]
    if k == "uf":
        return case["reps"] * case["atoms"]
    if k in ("forces", "grad") and case["form"] == "crystal":
        c = _cells(case)
        return 8 * c[0] * c[1] * c[2] - case["vac"]
    return case["atoms"]


def _host_arrays(n):
    """Page-locked host arrays for a whole batch's positions and velocities."""
    return [torch.empty((n, 3), dtype=torch.float64, pin_memory=True) for _ in range(2)]


def _static(case, seed):
    if case["form"] == "crystal":
        c = _cells(case)
        _, x, _, box = _crystal(*c, 700.0, _seed(seed, 1), case["vac"])
    else:
        x, box = _liquid(case["atoms"], _seed(seed, 1))
    return x, box


def prepare(case, seed):
    kind = case["kind"]
    prec = N.NEFE_FP64 if case.get("fp64") else N.NEFE_FP32
    if kind in ("fl", "io"):
        ctx = N.Context(precision=prec, dt=0.001, skin=case["skin"], nbr_cap=48)
        xs, vs = [], []
        for r in range(case["reps"]):
            r0, x, v, box = _crystal(*_cells(case), case["T"], _seed(seed, r), case.get("vac", 0))
            s = ctx.add_system(x, box, v=v, r0=r0, mass=MASS)
            ctx.set_thermostat(s, case["T"], 0.1, _seed(seed, r))
            ctx.set_schedule(s, N.NEFE_SCHED_FL, direction=1 if r % 2 == 0 else -1, nsteps=20000, k_E=5.0)
            xs.append(x)
            vs.append(v)
        st = {"ctx": ctx}
        if kind == "io":
            st["x"], st["v"] = _host_arrays(sum(len(x) for x in xs))
            st["x"].copy_(torch.from_numpy(np.concatenate(xs)))
            st["v"].copy_(torch.from_numpy(np.concatenate(vs)))
    elif kind == "dcci":
        ctx = N.Context(precision=prec, dt=0.001, skin=case["skin"], nbr_cap=48)
        pairs = []
        for k, n in enumerate(I.log_uniform_sizes(case["pairs"], case["lo"], case["hi"], seed=2021)):
            ids = []
            for q, (r0, box) in enumerate((I.diamond(*I.diamond_cells_for(n)), I.beta_tin(*I.beta_tin_cells_for(n)))):
                sd = _seed(seed, 2 * k + q)
                x = r0 + np.random.default_rng(sd).standard_normal(r0.shape) * math.sqrt(KB * 400.0 / 6.1)
                s = ctx.add_system(x, box, v=_velocities(len(x), 400.0, sd), mass=MASS)
                ctx.set_thermostat(s, 400.0, 0.1, sd)
                ctx.set_barostat(s, N.NEFE_BARO_ISO if q == 0 else N.NEFE_BARO_ANISO, 10.0, 0.5)
                ids.append(s)
            pairs.append(ctx.pair_dcci(ids[0], ids[1], 400.0, 10.0, N.NEFE_DCCI_PRESS, 10.0, 15.0, 100000))
        st = {"ctx": ctx, "pairs": pairs}
    elif kind == "rs":
        ctx = N.Context(precision=prec, dt=0.001, skin=case["skin"], nbr_cap=48)
        n = case["atoms"]
        for r in range(case["reps"]):
            for q in range(3):
                sd = _seed(seed, 3 * r + q)
                if q == 2:
                    x, box = _liquid(n, sd)
                else:      # the first n sites of a crystal that holds at least n: an odd count leaves vacancies
                    r0, box = _at_least(I.diamond, 8, n) if q == 0 else _at_least(I.beta_tin, 4, n)
                    x = r0[:n] + np.random.default_rng(sd).standard_normal((n, 3)) * math.sqrt(KB * 400.0 / 6.1)
                s = ctx.add_system(x, box, v=_velocities(n, 400.0, sd), mass=MASS)
                ctx.set_thermostat(s, 400.0, 0.1, sd)
                ctx.set_barostat(s, N.NEFE_BARO_ANISO if q == 1 else N.NEFE_BARO_ISO, case["P"], 1.0)
                ctx.set_schedule(s, N.NEFE_SCHED_RS, nsteps=50000, lambda_f=0.2, P_GPa=case["P"])
        st = {"ctx": ctx}
    elif kind == "uf":
        ctx = N.Context(precision=prec, dt=0.001, skin=case["skin"], nbr_cap=48)
        for r in range(case["reps"]):
            sd = _seed(seed, r)
            x, box = _liquid(case["atoms"], sd, 0.05225)
            s = ctx.add_system(x, box, v=_velocities(len(x), 2200.0, sd), mass=MASS)
            ctx.set_uf_params(s, N.uf_params(*UF))
            ctx.set_thermostat(s, 2200.0, 0.1, sd)
            ctx.set_schedule(s, N.NEFE_SCHED_FL, direction=1 if r % 2 == 0 else -1, nsteps=20000, ref=N.NEFE_REF_UF)
        st = {"ctx": ctx}
    elif kind == "adjoint":
        n, sd = case["atoms"], _seed(seed, 0)
        if case["sched"] == "rs":
            x, box = _liquid(n, sd)
            adj = N.Adjoint(x, _velocities(n, 1700.0, sd), box, kind=N.NEFE_SCHED_RS, lambda_f=0.5, T=1700.0, tdamp=0.1,
                            seed=sd, nsched=2000, checkpoint_every=case["every"])
        else:
            r0, box = _at_least(I.diamond, 8, n)
            x = r0[:n] + np.random.default_rng(sd).standard_normal((n, 3)) * math.sqrt(KB * 400.0 / 6.1)
            adj = N.Adjoint(x, _velocities(n, 400.0, sd), box, kind=N.NEFE_SCHED_FL, r0=r0[:n], k_E=5.0, T=400.0,
                            tdamp=0.1, seed=sd, nsched=1000, checkpoint_every=case["every"])
        return {"case": case, "adj": adj}
    else:
        x, box = _static(case, seed)
        n, rcs = len(x), 1.80 * 2.0951 + case["skin"]
        xd = torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
        if kind == "grad":
            theta = torch.tensor(AG.SILICON_THETA, dtype=torch.float64, requires_grad=True)
            return {"case": case, "x": xd.requires_grad_(True), "theta": theta, "box": box, "prec": prec}
        i32 = dict(dtype=torch.int32, device="cuda")
        f64 = dict(dtype=torch.float64, device="cuda")
        # rows past a row's length are the caller's: zeroed once, so that lists compare as a whole
        return {"case": case, "x": xd, "n": n, "box": box, "rcs": rcs, "prec": prec,
                "nbr": torch.zeros(n * 48, **i32), "cnt": torch.zeros(n, **i32), "f": torch.zeros(3 * n, **f64),
                "e": torch.zeros(n, **f64), "ev": torch.zeros(7, **f64), "prm": N.nefe_sw_params_silicon()}
    ctx.setup()
    if case.get("tune"):
        ctx.autotune()
    if kind != "io":
        st["x"], st["v"] = _host_arrays(sum(ctx.n))
    st["case"] = case
    return st


def _at_least(make, basis, n):
    """The smallest near-cubic crystal with at least n atoms (cells at least the list radius twice)."""
    if basis == 8:
        m = 2
        while 8 * m ** 3 < n:
            m += 1
        c = [m, m, m]
        while c[2] > 2 and 8 * c[0] * c[1] * (c[2] - 1) >= n:
            c[2] -= 1
    else:
        c = list(I.beta_tin_cells_for(max(n, 128)))
        while 4 * c[0] * c[1] * c[2] < n:
            c[2] += 1
    return make(*c)


# ------------------------------------------------------------------------------------- one pass
def _engine_outputs(ctx, x, v, fp64, state=True):
    ft = np.float64 if fp64 else np.float32
    res = ctx.results_all()
    out = {k: np.array([r[k] for r in res]).astype(ft) for k in ("W", "lambda", "U", "U_E", "K", "P", "V", "box", "dHdl", "H",
                                                                "mean_H", "mean_dHdl")}
    out["error"] = np.array([r["error"] for r in res], dtype=np.int64)
    if state:
        ctx.get_state_all(x.numpy(), v.numpy())
        out["x"], out["v"] = (x, v) if fp64 else (x.float(), v.float())
    return out


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("fl", "dcci", "rs", "uf"):
        ctx = st["ctx"]
        ctx.run(case["steps"])
        out = _engine_outputs(ctx, st["x"], st["v"], case.get("fp64", False))
        if kind == "dcci":
            out["pairs"] = np.array([ctx.pair(p)[:3] for p in st["pairs"]]).astype(np.float32)
        return out
    if kind == "io":
        ctx = st["ctx"]
        ctx.set_state_all(st["x"].numpy(), st["v"].numpy())
        ctx.run(case["steps"])
        return _engine_outputs(ctx, None, None, False, state=False)
    if kind == "adjoint":
        W = st["adj"].forward(case["steps"])
        g, gx, gv = st["adj"].backward(initial_state=True)
        return {"W": W, "g": g, "gx": gx, "gv": gv}
    if kind == "grad":
        E = AG.sw_energy(st["x"], st["theta"], st["box"], skin=case["skin"], precision=st["prec"])
        gx, gt = torch.autograd.grad(E, (st["x"], st["theta"]))
        return {"E": E.detach(), "gx": gx, "gtheta": gt} if case["fp64"] else \
            {"E": E.detach().float(), "gx": gx.float(), "gtheta": gt.float()}
    N.nefe_neighbor_build(st["x"], st["n"], st["box"], st["rcs"], 48, st["nbr"], st["cnt"])
    N.nefe_sw_forces(st["x"], st["n"], st["box"], st["rcs"], st["nbr"], st["cnt"], 48, st["prm"], st["prec"], st["f"],
                     st["e"], st["ev"])
    out = {"nbr": st["nbr"], "cnt": st["cnt"]}
    for k in ("f", "e", "ev"):
        out[k] = st[k] if case["fp64"] else st[k].float()
    return out


def work(case):
    """What one pass cannot do without.  An MD step reads and writes x and v, reads the sites and a
    Verlet row of about 28 entries and uses a force: 212 bytes and 600 operations an atom (the
    shell's pair and triplet terms through its moments).  An adjoint step is a forward step, its
    recomputation and a second-order product (three times a step's work in pairs of numbers)."""
    n, k = _atoms(case), case["kind"]
    if k in ("fl", "dcci", "rs", "uf"):
        flops = 600.0 + (3000.0 if k == "uf" else 0.0)       # ~110 reference-fluid pairs of ~27 operations
        return {"bytes": 212.0 * n * case["steps"], "flops": flops * n * case["steps"]}
    if k == "io":
        return {"bytes": 212.0 * n * case["steps"] + 48.0 * n, "flops": 600.0 * n * case["steps"]}
    if k == "adjoint":
        return {"bytes": 4 * 212.0 * n * case["steps"], "flops": 8 * 600.0 * n * case["steps"]}
    if k == "grad":
        return {"bytes": 48.0 * n, "flops": 900.0 * n}       # positions in, forces out
    return {"bytes": (24 + 48 * 4 + 4 + 24 + 8) * float(n), "flops": 600.0 * n}


# ----------------------------------------------------------------- the same results in 64 bits
THETA = (7.049556277, 0.6022245584, 4.0, 0.0, 1.80, 21.0, 1.20)
EPS, SIGMA, COS0 = 2.1683, 2.0951, -1.0 / 3.0


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _pairs(x, box, rc):
    """Every ordered pair (i, j) closer than rc (minimum image), sorted by (i, j).  x: (n, 3)."""
    n = len(x)
    nc = torch.floor(box / rc).to(torch.int64)
    if int(nc.min()) < 4 or n < (20000 if x.is_cuda else 4000):  # all pairs, in blocks of rows
        rows = max(1, 20_000_000 // n)
        got = []
        for a in range(0, n, rows):
            d = x[None, :, :] - x[a:a + rows, None, :]
            d -= box * torch.round(d / box)
            ii, jj = torch.nonzero((d * d).sum(-1) < rc * rc, as_tuple=True)
            ii = ii + a
            got.append(torch.stack([ii, jj])[:, ii != jj])
        return torch.cat(got, 1)
    w = x / box
    c = torch.minimum(((w - torch.floor(w)) * nc).to(torch.int64), nc - 1)
    cell = c[:, 0] + nc[0] * (c[:, 1] + nc[1] * c[:, 2])
    order = torch.argsort(cell, stable=True)
    ncell = int(nc.prod())
    count = torch.bincount(cell, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    occ = int(count.max())
    table = torch.full((ncell, occ), -1, dtype=torch.int64, device=x.device)
    cs = cell[order]
    table[cs, torch.arange(n, device=x.device) - start[cs]] = order
    got = []
    shifts = [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)]
    for s in shifts:
        o = (c + torch.tensor(s, device=x.device)) % nc
        t = table[o[:, 0] + nc[0] * (o[:, 1] + nc[1] * o[:, 2])]
        for q in range(occ):
            j = t[:, q]
            i = torch.nonzero(j >= 0)[:, 0]
            j = j[i]
            d = x[j] - x[i]
            d -= box * torch.round(d / box)
            keep = ((d * d).sum(1) < rc * rc) & (i != j)
            got.append(torch.stack([i[keep], j[keep]]))
    p = torch.cat(got, 1)
    return p[:, torch.argsort(p[0] * n + p[1])]


def _rows(p, n):
    """Pairs sorted by (i, j) as rows: neighbour table (n, m) padded with -1, and lengths."""
    cnt = torch.bincount(p[0], minlength=n)
    m = max(1, int(cnt.max()))
    start = torch.cumsum(cnt, 0) - cnt
    tab = torch.full((n, m), -1, dtype=torch.int64, device=p.device)
    tab[p[0], torch.arange(p.shape[1], device=p.device) - start[p[0]]] = p[1]
    return tab, cnt


def _sw_all(x, box, theta, blocks=200_000):
    """Energies per atom, forces, the virial and dE/dtheta.  x: (n, 3) float64."""
    n = len(x)
    tab, _ = _rows(_pairs(x, box, float(theta[4]) * SIGMA), n)
    x = x.clone().requires_grad_(True)
    strain = torch.zeros(3, 3, dtype=torch.float64, device=x.device, requires_grad=True)
    th = theta.clone().requires_grad_(True)
    e, gx, gs, gt = [], torch.zeros_like(x), torch.zeros_like(strain), torch.zeros_like(th)
    for a in range(0, n, blocks):
        t = tab[a:a + blocks]
        rows = torch.arange(a, a + len(t), device=x.device)
        tt = t.clamp(min=0)
        ok = t >= 0
        d = x[tt] - x[rows][:, None, :]
        d = d - box * torch.round(d / box).detach()
        d = d + d.detach() @ strain                          # d(d) = d strain: the virial is -dE/dstrain
        ei = _sw_d(d, ok, th)
        g = torch.autograd.grad(ei.sum(), (x, strain, th))
        gx, gs, gt = gx + g[0], gs + g[1], gt + g[2]
        e.append(ei.detach())
    return torch.cat(e), -gx, -gs, gt


def _sw_d(d, ok, theta):
    """Stillinger-Weber energy per atom (half of each pair, the triplets centred on the atom) from
    the vectors d (n, m, 3) to its neighbours; ok marks the entries in use."""
    A, B, p, q, a, lam, gam = theta
    d = torch.where(ok[..., None], d, torch.full_like(d, 10.0))
    r = (d * d).sum(-1).sqrt()
    s = r / SIGMA
    inn = ok & (s.detach() < a.detach() - 1e-12)
    sa = torch.where(inn, s, torch.full_like(s, 1.0))
    id_ = 1.0 / (sa - a)
    zero = torch.zeros_like(s)
    phi = torch.where(inn, EPS * A * (B * sa ** (-p) - sa ** (-q)) * torch.exp(id_), zero)
    g = torch.where(inn, torch.exp(gam * id_), zero)
    u = d / r[..., None]
    c = torch.einsum("iak,ibk->iab", u, u) - COS0
    h = EPS * lam * g[:, :, None] * g[:, None, :] * c * c
    h = h * (1.0 - torch.eye(h.shape[1], dtype=h.dtype, device=h.device))
    return 0.5 * phi.sum(1) + 0.5 * h.sum((1, 2))


def _mulhilo(m, b):
    """High and low 64 bits of m * b (numpy uint64 arrays), by 32-bit halves."""
    lo32 = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    a0, a1 = m & lo32, m >> s
    b0, b1 = b & lo32, b >> s
    t = a0 * b0
    k = a1 * b0 + (t >> s)
    w = a0 * b1 + (k & lo32)
    return a1 * b1 + (k >> s) + (w >> s), m * b


def _noise(seed, system, step, n, bits):
    """Thermostat normals (n, 3): Philox4x64-10 at counter (step, atom, system, 0), key (seed, 0),
    two Box-Muller pairs; uniforms of the top `bits` bits (24 in FP32 runs, 53 in FP64 runs)."""
    with np.errstate(over="ignore"):
        c = [np.full(n, step, dtype=np.uint64), np.arange(n, dtype=np.uint64), np.full(n, system, dtype=np.uint64),
             np.zeros(n, dtype=np.uint64)]
        k0, k1 = np.uint64(seed), np.uint64(0)
        for _ in range(10):
            h0, l0 = _mulhilo(np.uint64(0xD2E7470EE14C6C93), c[0])
            h1, l1 = _mulhilo(np.uint64(0xCA5A826395121157), c[2])
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
    u = [((v >> np.uint64(64 - bits)).astype(np.float64) + 0.5) * 2.0 ** -bits for v in c]
    r0, r1 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    return np.stack([r0 * np.cos(2 * np.pi * u[1]), r0 * np.sin(2 * np.pi * u[1]), r1 * np.cos(2 * np.pi * u[3])], 1)


def _fl_lambda(k, nsteps, direction):
    t = min(k / nsteps, 1.0)
    t = t if direction > 0 else 1.0 - t
    return t ** 5 * (70 * t ** 4 - 315 * t ** 3 + 540 * t ** 2 - 420 * t + 126)


def _fl_exact(case, seed):
    """The Frenkel-Ladd run in 64 bits: the Langevin velocity-Verlet step, left-point work."""
    dev, T, dt, kE, K = _dev(), case["T"], 0.001, 5.0, case["steps"]
    bits = 53 if case["fp64"] else 24
    me = MASS * MVV2E
    c, gam, amp = 0.5 * dt / me, me / 0.1, math.sqrt(2.0 * me * KB * T / (0.1 * dt))
    theta = torch.tensor(THETA, dtype=torch.float64, device=dev)
    out = {k: [] for k in ("W", "lambda", "U", "U_E", "K", "P", "V", "box", "dHdl", "H", "mean_H", "mean_dHdl")}
    xs, vs = [], []
    for r in range(case["reps"]):
        r0, x, v, box_ = _crystal(*_cells(case), T, _seed(seed, r), case["vac"])
        direction = 1 if r % 2 == 0 else -1
        r0, x, v, box = (torch.from_numpy(np.ascontiguousarray(t)).to(dev) for t in (r0, x, v, box_))
        n = len(x)
        V = float(box.prod())
        W = sumH = sumD = 0.0
        lam = _fl_lambda(0, 20000, direction)
        F = None
        for k in range(K + 1):
            if k > 0:
                v = v + c * F
                x = x + dt * v
            e, f, vir, _ = _sw_all(x, box, theta)
            d = x - r0
            xi = torch.from_numpy(_noise(_seed(seed, r), r, k, n, bits)).to(dev)
            F = (1.0 - lam) * f - lam * kE * d - gam * v + amp * (xi - xi.mean(0))
            if k > 0:
                v = v + c * F
            U, UE = float(e.sum()), float(0.5 * kE * (d * d).sum())
            kt = me * (v.T @ v)
            D, Kin = UE - U, 0.5 * float(torch.diagonal(kt).sum())
            H = Kin + (1.0 - lam) * U + lam * UE
            if k < K:
                nxt = _fl_lambda(k + 1, 20000, direction)
                W += D * (nxt - lam)
                sumH, sumD, lam = sumH + H, sumD + D, nxt
        P = (kt + (1.0 - lam) * vir) / V * GPA
        P = [float(P[a, b]) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
        for key, val in (("W", W), ("lambda", lam), ("U", U), ("U_E", UE), ("K", Kin), ("P", P), ("V", V),
                         ("box", box_), ("dHdl", D), ("H", H), ("mean_H", sumH / K), ("mean_dHdl", sumD / K)):
            out[key].append(val)
        xs.append(x.cpu())
        vs.append(v.cpu())
    out = {k: np.array(v) for k, v in out.items()}
    out["error"] = None
    out["x"], out["v"] = torch.cat(xs), torch.cat(vs)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "fl" and _atoms(case) * case["steps"] <= 3_000_000 and case["reps"] * case["steps"] <= 600:
        return _fl_exact(case, seed)
    if kind not in ("forces", "grad"):
        # long trajectories of many atoms, under a barostat or with the reference fluid, and the
        # gradient through one: minutes in plain torch
        return None
    dev = _dev()
    x, box = _static(case, seed)
    x, box = torch.from_numpy(x).to(dev), torch.from_numpy(box).to(dev)
    e, f, vir, gt = _sw_all(x, box, torch.tensor(THETA, dtype=torch.float64, device=dev))
    if kind == "grad":
        return {"E": e.sum(), "gx": -f.T.contiguous(), "gtheta": gt.cpu()}
    ev = torch.stack([e.sum()] + [vir[a, b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
    return {"nbr": None, "cnt": None, "f": f.T.contiguous().reshape(-1), "e": e, "ev": ev}
