"""Performance cases of the track stepper: what a program asks of it, through
``paper_0810_4737_gb300.reed``.

A case is one call that a program makes and waits for: a batch of ion tracks
with its range profile and per-track records (``Reed.run``), an adaptive
rare-event batch, one step of a parameter fit (``ProfileFunction``: the
differentiable profile and its gradient), or one force evaluation
(``Reed.forces``).  Workloads are those of ``workloads.py``; energies and
counts are theirs or smaller ones of the same kind, so that the calls range
from a handful of ions, where only the time of one step matters, to batches
that keep the whole GPU busy.  Two long workloads (CeO2 at 30 keV, 85 MeV
fission fragments) are cut after a given number of steps per track
(``step_cap``), as a trial run does.

A track's records and its contribution to the profile do not depend on
timing, so a call gives the same numbers whenever it is repeated; the records
come in the order in which the tracks finished and are sorted by track id
here.
"""
import math

import numpy as np
import torch

from paper_0810_4737_gb300 import reed
from paper_0810_4737_gb300.workloads import workload

B_SMALL = "b1kev_si_0k_zbl"
B_REED = "b50kev_si_300k_reed"
B_FIT = "b10kev_si_300k_adjoint"
AS_SI = "as10kev_si_300k_tersoff"
AR_CEO2 = "ar30kev_ceo2_300k_buck"
U_UO2 = "u85kev_uo2_300k_recoil"
KR_UO2 = "kr85mev_uo2_300k_recoil"

# Mean track of each workload, in steps: reference
# energy (eV), steps of a primary at that energy, growth with the energy.
STEPS = {B_SMALL: (1e3, 3000, 0.72), B_REED: (1e4, 16600, 0.74), B_FIT: (1e4, 16600, 0.74), AS_SI: (1e4, 4700, 0.4),
         AR_CEO2: (3e3, 3600, 0.39), U_UO2: (8.5e4, 5800, 0.33), KR_UO2: (1e6, 100000, 0.8)}
# Operations of one step that no implementation can leave out: ion-target
# pairs inside the cutoff (35 each), moving atoms (24 each), Tersoff
# bond-angle terms (60 each), target-target pairs (45 each).
STEP_FLOPS = {B_SMALL: 25 * 35 + 50 * 24, B_REED: 26 * 35 + 52 * 24, B_FIT: 26 * 35 + 52 * 24,
              AS_SI: 25 * 35 + 211 * 24 + 4360 * 60, AR_CEO2: 33 * 35 + 740 * 24 + 10000 * 45,
              U_UO2: 37 * 35 + 74 * 24, KR_UO2: 39 * 35 + 78 * 24}

# Records that an adaptive batch keeps room for, per primary (12 cloning
# depths make some 60 tracks of a primary, in heavy-tailed numbers).
RECORDS = 400


def _tracks(name, w, ions, energy, precision="mixed", **more):
    return dict({"name": name, "kind": "tracks", "workload": w, "ions": ions, "energy": float(energy),
                 "precision": precision, "adaptive": False, "epoch": 0, "step_cap": 0}, **more)


def listed():
    return [
        # the smallest batch of the repository: 32 boron ions, a look at a new
        # target or energy; a few tracks on an otherwise idle GPU
        _tracks("b_few", B_SMALL, 32, 1000.0),
        # a boron implant profile at room temperature: thousands of ions, the
        # plain throughput of the ion-target model
        _tracks("b_profile", B_REED, 3001, 10000.0),
        # the same model in plain FP64, the check of a mixed-form profile
        _tracks("b_fp64", B_SMALL, 500, 1000.0, precision="fp64"),
        # deep tails of a channelled profile: adaptive cloning depths, weights
        # 2^-k, clones handed to idle CTAs
        _tracks("b_deep_adaptive", B_REED, 150, 20000.0, adaptive=True, epoch=64),
        # arsenic with Tersoff target forces: a few low-energy ions
        _tracks("as_few", AS_SI, 37, 2000.0),
        # ... and the full batch of the benchmark
        _tracks("as_batch", AS_SI, 4096, 10000.0),
        # ... and a low-energy batch in plain FP64
        _tracks("as_fp64", AS_SI, 61, 100.0, precision="fp64"),
        # argon into ceria: Buckingham target forces and the damage map, the
        # first 2000 steps of each track
        _tracks("ar_ceo2", AR_CEO2, 203, 30000.0, step_cap=2000),
        # uranium recoils in bulk UO2 with adaptive cloning distances
        _tracks("u_recoils", U_UO2, 512, 85000.0, adaptive=True, epoch=256),
        # 85 MeV fission fragments with the energy term of the time step, the
        # first 10000 steps of each track: fewer tracks than the GPU has room for
        _tracks("kr_mev", KR_UO2, 131, 85.0e6, step_cap=10000),
        # one step of a fit of the stopping and the screening correction to a
        # measured profile: profile and gradient
        {"name": "fit_step", "kind": "fit", "workload": B_FIT, "ions": 1024, "energy": 5000.0, "precision": "mixed"},
        # forces of one thermal configuration, ion included
        {"name": "forces_si", "kind": "forces", "workload": AS_SI, "cells": 4, "precision": "mixed"},
    ]


def _between(rng, lo, hi):
    """A whole number, spread over the logarithm of its range, odd or even."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice([B_SMALL, B_REED, AS_SI, AS_SI, AR_CEO2, U_UO2, KR_UO2, "fit", "forces"])
    fp64 = rng.random() < 0.25
    p = "fp64" if fp64 else "mixed"
    if family == "forces":
        w = rng.choice([B_SMALL, AS_SI, AR_CEO2])
        # (four cells of Tersoff lists in FP64 are more than an SM's shared memory)
        cells = [3, 4] if w == AR_CEO2 else ([2, 3] if w == AS_SI and fp64 else [2, 3, 4])
        return {"kind": "forces", "workload": w, "cells": rng.choice(cells), "precision": p}
    if family == "fit":
        return {"kind": "fit", "workload": B_FIT, "ions": _between(rng, 16, 128 if fp64 else 2048),
                "energy": float(_between(rng, 500, 1500 if fp64 else 10000)), "precision": p}
    c = _tracks("", family, 0, 0.0, precision=p)
    del c["name"]
    if family == B_SMALL:
        c["ions"], c["energy"] = _between(rng, 1, 700 if fp64 else 8192), float(_between(rng, 200, 1500))
    elif family == B_REED:
        c["energy"] = float(_between(rng, 1000, 2000 if fp64 else 20000))
        c["ions"] = _between(rng, 16, 256 if fp64 else 4096)
        if not fp64 and rng.random() < 0.5:
            c["adaptive"], c["epoch"], c["ions"] = True, _between(rng, 32, 128), _between(rng, 64, 150)
    elif family == AS_SI:
        c["ions"], c["energy"] = _between(rng, 1, 152 if fp64 else 2500), float(_between(rng, 100, 150 if fp64 else 10000))
    elif family == AR_CEO2:
        c["energy"] = float(_between(rng, 300, 30000))
        c["ions"], c["step_cap"] = _between(rng, 1, 76 if fp64 else 304), _between(rng, 50, 200 if fp64 else 2000)
    elif family == U_UO2:
        c["energy"] = float(_between(rng, 1000, 2000 if fp64 else 85000))
        c["ions"] = _between(rng, 8, 128 if fp64 else 3000)
        if not fp64 and rng.random() < 0.5:
            c["adaptive"], c["epoch"], c["ions"] = True, _between(rng, 64, 512), _between(rng, 64, 700)
    else:
        c["energy"] = float(_between(rng, 1e6, 85e6))
        c["ions"], c["step_cap"] = _between(rng, 1, 300), _between(rng, 500, 1500 if fp64 else 20000)
    return c


def _precision(case):
    return reed.PREC_FP64 if case["precision"] == "fp64" else reed.PREC_MIXED


# the point of a fit at which the profile and its gradient are taken: a
# little off the default stopping, with some local density in the drag and a
# small screening correction
THETA = [1.05, 0.1, 0.02, -0.01, 0.03, 0.0, 0.01, -0.02]


def _configuration(case, seed):
    """A thermal block of crystal and an ion somewhere inside it."""
    w = workload(case["workload"], n=case["cells"], margin=0)
    rng = np.random.default_rng(seed)
    if w["lattice"] == "diamond":
        basis = [(0, 0, 0), (0, .5, .5), (.5, 0, .5), (.5, .5, 0), (.25, .25, .25), (.25, .75, .75), (.75, .25, .75),
                 (.75, .75, .25)]
        species = [0] * 8
    else:
        basis = [(0, 0, 0), (0, .5, .5), (.5, 0, .5), (.5, .5, 0)]
        basis += [(x, y, z) for x in (.25, .75) for y in (.25, .75) for z in (.25, .75)]
        species = [0] * 4 + [1] * 8
    m = case["cells"]
    cells = np.array([(i, j, k) for i in range(m) for j in range(m) for k in range(m)], dtype=float) - m // 2
    xyz = (cells[:, None, :] + np.array(basis)[None, :, :]).reshape(-1, 3) * w["a"]
    xyz += rng.normal(scale=0.076, size=xyz.shape)
    sp = np.tile(np.array(species, dtype=np.int32), cells.shape[0])
    # the ion keeps 0.6 A from the nearest atom
    while True:
        ion = rng.uniform(-0.4, 0.4, size=3) * w["a"]
        if np.min(np.linalg.norm(xyz - ion, axis=1)) > 0.6:
            return w, ion, xyz, sp


def prepare(case, seed):
    if case["kind"] == "forces":
        w, ion, xyz, sp = _configuration(case, seed)
        return {"case": case, "ctx": reed.Reed(w), "ion": ion, "xyz": xyz, "sp": sp}
    w = workload(case["workload"], energy=case["energy"])
    if case["kind"] == "fit":
        fn, holder = reed.ProfileFunction.make(w, case["ions"], seed, 10.0, int(w["n_bins"]), float(w["bin_w"]),
                                               precision=_precision(case))
        theta = torch.tensor(THETA, dtype=torch.float64, device="cuda", requires_grad=True)
        g = torch.Generator().manual_seed(seed)
        target = torch.rand(int(w["n_bins"]), generator=g, dtype=torch.float64).cuda() / (w["n_bins"] * w["bin_w"])
        return {"case": case, "fn": fn, "holder": holder, "theta": theta, "target": target}
    if case["step_cap"]:
        w["step_cap"] = case["step_cap"]
    if not case["adaptive"]:
        w["thresholds"] = []
    return {"case": case, "ctx": reed.Reed(w), "seed": seed}


def run(state):
    case = state["case"]
    if case["kind"] == "forces":
        e, f_ion, f_atoms, rho = state["ctx"].forces(state["ion"], state["xyz"], state["sp"], precision=_precision(case))
        return {"energy": e, "f_ion": f_ion, "f_atoms": f_atoms, "rho": rho}
    if case["kind"] == "fit":
        theta = state["theta"]
        theta.grad = None
        p = state["fn"](theta)
        loss = (1e4 * (p - state["target"])).square().sum()
        loss.backward()
        return {"profile": p.detach(), "grad": theta.grad}
    ctx = state["ctx"]
    ctx.reset()
    more = {}
    if case["adaptive"]:
        more = {"adaptive": True, "n_initial": 50, "epoch_size": case["epoch"], "record_capacity": RECORDS * case["ions"]}
    ctx.run(n_ions=case["ions"], seed=state["seed"], precision=_precision(case), **more)
    bins, extra = ctx.profile()
    rec = ctx.records()
    rec = rec[np.argsort(rec["id"], kind="stable")]
    if case["adaptive"]:   # the number of clones depends on the tracks: fill up to the size of the record buffer
        full = np.zeros(RECORDS * case["ions"], dtype=rec.dtype)
        full[:len(rec)] = rec
        rec = full
    out = {"bins": bins, "extra": extra, "id": rec["id"].view(np.int64), "z": rec["z"].copy(), "t": rec["t"].copy(),
           "steps": rec["steps"].copy(), "level": rec["level"].copy(), "status": rec["status"].copy()}
    if case["adaptive"]:
        out["depths"] = ctx.thresholds()
    if ctx.w["damage_n"]:
        out["damage"], out["damage_outside"] = ctx.damage_map()
    return out


def work(case):
    name = case["workload"]
    if case["kind"] == "forces":
        w = workload(name)
        n = (8 if w["lattice"] == "diamond" else 12) * case["cells"] ** 3
        flops = 30 * 35 + n * {"none": 0, "tersoff": 12 * 60, "buckingham": 25 * 45}[w["tt"]]
        return {"bytes": n * (24 + 4 + 24) + 64, "flops": flops}
    w = workload(name)
    e0, steps, power = STEPS[name]
    steps *= (case["energy"] / e0) ** power
    if case.get("step_cap"):
        steps = min(steps, case["step_cap"])
    tracks = case["ions"]
    if case.get("adaptive"):   # clones: about half a track per depth and primary after the first 50
        tracks += 0.5 * len(w["thresholds"]) * max(0, case["ions"] - 50)
    flops = tracks * steps * STEP_FLOPS[name]
    if case["kind"] == "fit":   # the last 200 steps forward again and backward, and the kernel-density profile
        flops += tracks * (200 * 4 * STEP_FLOPS[name] + 2 * 20 * w["n_bins"])
        return {"bytes": tracks * (48 + 64) + 2 * 8 * w["n_bins"], "flops": flops}
    return {"bytes": tracks * 48 + 8 * (w["n_bins"] + 3) + 8 * w["damage_n"] ** 3, "flops": flops}


# ---- one configuration's energy and forces in 64 bits ----------------------

def _taper(r, lo, hi):
    """1 below lo, 0 above hi, a C2 quintic in between."""
    t = ((r - lo) / (hi - lo)).clamp(0.0, 1.0)
    return 1.0 - t ** 3 * (10.0 - 15.0 * t + 6.0 * t * t)


def _zbl(r, z1, z2):
    x = r * (z1 ** 0.23 + z2 ** 0.23) / (0.8854 * 0.529177)
    phi = (0.18175 * torch.exp(-3.1998 * x) + 0.50986 * torch.exp(-0.94229 * x) + 0.28022 * torch.exp(-0.4029 * x)
           + 0.02817 * torch.exp(-0.20162 * x))
    return z1 * z2 * 14.399645 / r * phi


def _pairs(x, cut):
    """Every ordered pair of atoms closer than cut: indices and vectors."""
    d2 = (x.detach()[:, None, :] - x.detach()[None, :, :]).square().sum(-1)
    d2.fill_diagonal_(math.inf)
    i, j = torch.nonzero(d2 < cut * cut, as_tuple=True)
    return i, j


def _tersoff(w, x, z):
    t = w["tersoff"]
    cut = t["R"] + t["D"]
    i, j = _pairs(x, cut)
    d = x[j] - x[i]
    r = d.norm(dim=1)
    fc = torch.where(r < t["R"] - t["D"], torch.ones_like(r), 0.5 - 0.5 * torch.sin(0.5 * math.pi * (r - t["R"]) / t["D"]))
    # bonds (i, j) and (i, k) with the same centre: all pairs of rows of i's block
    same = (i[:, None] == i[None, :]) & (torch.arange(len(i))[:, None] != torch.arange(len(i))[None, :])
    p, q = torch.nonzero(same, as_tuple=True)
    u = d / r[:, None]
    cos = (u[p] * u[q]).sum(1)
    c2, d2 = t["c"] ** 2, t["d"] ** 2
    s = (t["h"] - cos).square()
    g = 1.0 + c2 / d2 * s / (d2 + s)
    zeta = torch.zeros_like(r).index_add(0, p, fc[q] * g)
    bond = (1.0 + (t["beta"] * zeta).pow(t["n"])).pow(-0.5 / t["n"])
    v = fc * (t["A"] * torch.exp(-t["lam1"] * r) - bond * t["B"] * torch.exp(-t["lam2"] * r))
    b = _taper(r, *w["blend"])
    return 0.5 * ((1.0 - b) * v + b * _zbl(r, z, z)).sum()


def _buckingham(w, x, sp):
    k = w["buckingham"]
    a, rho, c = (torch.tensor(k[n], dtype=torch.float64) for n in ("A", "rho", "C"))
    zs = torch.tensor([s["Z"] for s in w["species"]], dtype=torch.float64)
    i, j = _pairs(x, w["buck_cut"][1])
    r = (x[j] - x[i]).norm(dim=1)
    t = sp[i] + sp[j]
    v = a[t] * torch.exp(-r / rho[t]) - c[t] / r ** 6
    b = _taper(r, *w["buck_blend"])
    v = (1.0 - b) * v + b * _zbl(r, zs[sp[i]], zs[sp[j]])
    return 0.5 * (v * _taper(r, *w["buck_cut"])).sum()


def exact(case, seed):
    """The forces of one configuration, from its energy.  Whole tracks have no
    64-bit value to be held against: a rounding difference grows without
    bound along a track, and a track in 64 bits by plain array operations
    takes minutes."""
    if case["kind"] != "forces":
        return None
    w, ion, xyz, sp = _configuration(case, seed)
    xi = torch.tensor(ion, dtype=torch.float64, requires_grad=True)
    x = torch.tensor(xyz, dtype=torch.float64, requires_grad=True)
    s = torch.tensor(sp, dtype=torch.int64)
    zs = torch.tensor([q["Z"] for q in w["species"]], dtype=torch.float64)
    r = (x - xi).norm(dim=1)
    near = torch.nonzero(r.detach() < w["rc"]).flatten()
    e = (_zbl(r[near], w["ion"]["Z"], zs[s[near]]) * _taper(r[near], w["rt"], w["rc"])).sum()
    if w["tt"] == "tersoff":
        e = e + _tersoff(w, x, w["species"][0]["Z"])
    elif w["tt"] == "buckingham":
        e = e + _buckingham(w, x, s)
    g_ion, g = torch.autograd.grad(e, (xi, x))
    return {"energy": float(e.detach()), "f_ion": (-g_ion).numpy(), "f_atoms": (-g).numpy(), "rho": None}
