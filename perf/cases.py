"""What a user of the library has it do, as cases that can be timed and checked.

The work is the force-field evaluation and what is built on it: one energy / force / virial evaluation of a
box handed over by an MD engine (`DPModel.compute`), velocity-Verlet MD inside the library (`DPModel.verlet`),
MD of many boxes at once (`DPModel.md_run_batch`), labelling many boxes at once (`DPModel.compute_batch`) and the
gradient step of a training loop (`ParamLoss`).  Systems, sizes, time step and models are those of the benchmark
and the tests: water (r_c 6 A, sel 46/92) from 64 molecules to 4096, FCC copper (r_c 8 A, sel 512) up to 131,072
atoms, 0.5 fs, a list rebuild every 10 steps.  Single evaluations and training use the models with environment
statistics and trained-size forces, MD the plain ones (the others are no stable potentials), as the benchmark does.

A model of FP32 or mixed precision computes energies, forces and gradients in FP32 sums, which the library
hands over in FP64 arrays; a program with such a model keeps them in FP32 (its own data type), and so does run().
Positions and velocities are FP64 state in every precision.
"""
import json
import math
import os

import numpy as np
import torch

import paper_2410_22867_gb300 as dp
from paper_2410_22867_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(dp.__file__)))
KAPPA = 9.648533e-3  # A fs^-2 per eV A^-1 amu^-1
DT = 0.5             # fs
EVERY = 10           # steps between list rebuilds


def listed():
    return [
        # latency-bound MD of a small box, the case behind ns/day figures
        {"name": "md_water64_fp16", "kind": "md", "system": "water", "size": 64, "precision": "mix_fp16", "steps": 10},
        # reference-quality evaluation of a small box (validation of a model, phonons, relaxations)
        {"name": "compute_water64_fp64", "kind": "compute", "system": "water", "size": 64, "precision": "fp64"},
        # the precision between: one evaluation of a mid-size box for a host MD engine; odd size
        {"name": "compute_water777_fp32", "kind": "compute", "system": "water", "size": 777, "precision": "fp32"},
        # a sheared (triclinic) box in bf16, ragged size
        {"name": "compute_water1500_tri_bf16", "kind": "compute", "system": "water", "size": 1500, "precision": "mix_bf16",
         "shear": 0.12},
        # production MD of liquid water, 12,288 atoms
        {"name": "md_water4096_fp16", "kind": "md", "system": "water", "size": 4096, "precision": "mix_fp16", "steps": 10},
        # many small boxes in one MD run (sampling, active learning)
        {"name": "md_batch64_fp16", "kind": "batch_md", "system": "water", "size": 64, "precision": "mix_fp16", "steps": 10},
        # the FP64 evaluation that mixed precision is validated against, on the 4,000-atom copper box
        {"name": "compute_cu10_fp64", "kind": "compute", "system": "copper", "size": 10, "precision": "fp64"},
        # FP32 evaluation of a 32,000-atom crystal
        {"name": "compute_cu20_fp32", "kind": "compute", "system": "copper", "size": 20, "precision": "fp32"},
        # the compressed (tabulated) model on the same crystal
        {"name": "compute_cu20_table_fp16", "kind": "compute", "system": "copper", "size": 20, "precision": "mix_fp16",
         "table": 256},
        # one call per step from a host MD engine on the benchmark's 131,072-atom crystal
        {"name": "compute_cu32_fp16", "kind": "compute", "system": "copper", "size": 32, "precision": "mix_fp16"},
        # the benchmark itself: NVE MD of 131,072 atoms
        {"name": "md_cu32_fp16", "kind": "md", "system": "copper", "size": 32, "precision": "mix_fp16", "steps": 10},
        # a training step on one 3,072-atom frame (loss and its gradient for every parameter)
        {"name": "train_water1024_fp32", "kind": "train", "system": "water", "size": 1024, "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Kinds, systems, precisions and sizes of the ranges of listed(); upper ends per precision as there."""
    kind = rng.choice(["compute", "compute", "compute", "md", "md", "batch", "train"])
    prec = rng.choice(["fp64", "fp32", "mix_bf16", "mix_fp16", "mix_fp16"])
    if kind == "train":
        prec = rng.choice(["fp64", "fp32", "fp32"])
        return {"kind": kind, "system": "water", "size": _log(rng, 32, 96 if prec == "fp64" else 1024), "precision": prec}
    if kind == "batch":
        md = rng.random() < 0.5
        if md:
            prec = rng.choice(["mix_bf16", "mix_fp16"])
            return {"kind": "batch_md", "system": "water", "size": _log(rng, 3, 64), "precision": prec, "steps": EVERY}
        return {"kind": "batch_compute", "system": "water", "size": _log(rng, 3, 6 if prec == "fp64" else 64),
                "precision": prec}
    system = rng.choice(["water", "copper"])
    if kind == "md":
        prec = rng.choice(["fp32", "mix_bf16", "mix_fp16", "mix_fp16"])
        hi = {"water": 512 if prec == "fp32" else 4096, "copper": 8 if prec == "fp32" else 32}[system]
        return {"kind": kind, "system": system, "size": _log(rng, 64 if system == "water" else 6, hi),
                "precision": prec, "steps": EVERY}
    hi = {"water": {"fp64": 512}.get(prec, 4096), "copper": {"fp64": 10, "fp32": 20}.get(prec, 32)}[system]
    case = {"kind": kind, "system": system, "size": _log(rng, 64 if system == "water" else 6, hi), "precision": prec}
    if rng.random() < 0.25:
        case["shear"] = round(rng.uniform(0.02, 0.15), 3)
    if rng.random() < 0.2:
        if system == "copper" and prec != "fp64":
            case["size"] = min(case["size"], 20)
        case["table"] = 256
    return case


# ------------------------------------------------------------------ inputs
def _weights(case):
    if case["kind"] in ("md", "batch_md"):
        return synth.water_weights(1001) if case["system"] == "water" else synth.copper_weights(1001)
    with open(os.path.join(ROOT, "tests", "golden", "env_stats.json")) as f:
        return synth.normalised_weights(case["system"], json.load(f))


def _systems(case, seed):
    """The boxes of a case: one, or `size` replicas of 32 to 2048 molecules (log-uniform counts that belong to the
    case, densities and configurations from the seed)."""
    if case["kind"].startswith("batch"):
        counts = np.random.default_rng(case["size"]).uniform(math.log(32), math.log(2048), case["size"])
        rng = np.random.default_rng(seed)
        return [synth.water_box(int(round(math.exp(c))), int(rng.integers(2 ** 31 - 1)), density=float(1.0 + rng.uniform(-0.03, 0.03)))
                for c in counts]
    s = synth.water_box(case["size"], seed) if case["system"] == "water" else synth.copper_fcc(case["size"], seed)
    g = case.get("shear", 0.0)
    if g:  # the same box under a volume-keeping shear
        m = np.array([[1.0, 0.0, 0.0], [g, 1.0, 0.0], [-0.5 * g, 0.7 * g, 1.0]])
        s.coords = s.coords @ m
        s.box = (s.box.reshape(3, 3) @ m).reshape(-1)
    return [s]


def _inputs(case, seed):
    """Host arrays that a program has in hand: coordinates, types, offsets, boxes, velocities, labels."""
    systems = _systems(case, seed)
    coords, types, offs, boxes = synth.concat(systems)
    h = {"x": coords, "types": types, "offs": offs, "boxes": boxes, "masses": systems[0].masses()}
    if case["kind"] in ("md", "batch_md"):
        h["v"] = np.concatenate([synth.maxwell_boltzmann(h["masses"][s.types], 300.0, seed + 7 + k)
                                 for k, s in enumerate(systems)])
    if case["kind"] == "train":
        rng = np.random.default_rng(seed + 11)
        n = len(types)
        h["E0"] = float(rng.normal(0.0, 0.1)) * n
        h["F0"] = rng.normal(0.0, 0.5, size=(n, 3))
        h["cE"], h["cF"] = 1.0 / n ** 2, 1.0 / (3 * n)  # per-atom energy error, mean square force error
    return h


def prepare(case, seed):
    h = _inputs(case, seed)
    w = _weights(case)
    n = len(h["types"])
    model = dp.DPModel(w, case["precision"], max_atoms=n, max_replicas=len(h["offs"]) - 1)
    if case.get("table"):
        model.tabulate(case["table"])
    s = {"case": case, "model": model, "box": h["boxes"][0], "boxes": h["boxes"], "offs": h["offs"],
         "x0": torch.tensor(h["x"], device="cuda"), "types": torch.tensor(h["types"], device="cuda")}
    if "v" in h:
        s["v0"] = torch.tensor(h["v"], device="cuda")
        s["x"], s["v"] = s["x0"].clone(), s["v0"].clone()
        s["md"] = model.md_state(s["x"], s["v"], s["types"], h["boxes"], h["masses"],
                                 atom_offsets=h["offs"] if case["kind"] == "batch_md" else None, rebuild_every=EVERY)
    if case["kind"] == "train":
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        s["theta"] = torch.tensor(w.theta, dtype=dtype, device="cuda", requires_grad=True)
        s.update(F0=torch.tensor(h["F0"], device="cuda"), E0=h["E0"], cE=h["cE"], cF=h["cF"])
    return s


def run(s):
    case, model = s["case"], s["model"]
    kind = case["kind"]
    if kind == "train":
        theta = s["theta"]
        theta.grad = None
        loss = dp.ParamLoss.apply(theta, model, s["x0"], s["types"], s["box"], s["E0"], s["F0"], s["cE"], s["cF"])
        loss.backward()
        return {"loss": loss.detach(), "grad": theta.grad}
    if kind == "compute":
        out = model.compute(s["x0"], s["types"], s["box"])
    elif kind == "batch_compute":
        out = model.compute_batch(s["x0"], s["types"], s["offs"], s["boxes"])
    else:
        s["x"].copy_(s["x0"])  # the run starts from the same state in every pass
        s["v"].copy_(s["v0"])
        s["md"].step = 0
        if kind == "md":
            k = model.verlet(s["md"], DT, case["steps"])
        else:
            k = model.md_run_batch(s["md"], DT, case["steps"])
        out = {q: k[q] for q in ("forces", "potential", "kinetic", "virial")}
    if case["precision"] != "fp64":
        out = {q: t.float() for q, t in out.items()}
    if kind in ("md", "batch_md"):
        out.update(x=s["x"], v=s["v"])
    return out


# ------------------------------------------------------------------ work
def _rows(case):
    """(atoms, neighbour rows within r_c) of a case, from the densities."""
    if case["system"] == "copper":
        n = 4 * case["size"] ** 3
        return n, n * (4.0 / 3.0 * math.pi * 8.0 ** 3 * 4.0 / 3.634 ** 3)
    mol = case["size"] * (485.0 if case["kind"].startswith("batch") else 1.0)
    per_a3 = synth.AVOGADRO_PER_A3 / synth.WATER_G_PER_MOL
    return int(3 * mol), 3 * mol * 4.0 / 3.0 * math.pi * 6.0 ** 3 * 3 * per_a3


def work(case):
    """Operations without any recomputation: embedding net forward 6,275 and backward 6,275 multiply-adds a neighbour,
    400 for T and 800 for dE/dT against G and R_hat; fitting net 499,440 forward and as many backward an atom.
    Bytes: positions and types in, energies, forces (and MD state) out, the parameters once.  A training step carries a
    tangent beside every forward value and goes back through both, with weight gradients."""
    n, rows = _rows(case)
    flops = 2.0 * (rows * (6275 + 400 + 6275 + 800) + n * 2 * 499440)
    types = 2 if case["system"] == "water" else 1
    weights = (types * types * 6450 + types * 500161) * 8.0
    steps = case.get("steps", 0)
    if case["kind"] == "train":
        return {"flops": 2.0 * (rows * (2 * 6275 + 800) * 3 + n * 2 * 499440 * 3), "bytes": 2 * weights + n * (24 + 4 + 24.0)}
    if steps:
        return {"flops": flops * (steps + 1), "bytes": weights + n * (4 * 24 + 4 + 24.0)}
    return {"flops": flops, "bytes": weights + n * (24 + 4 + 8 + 24.0)}


# ------------------------------------------------------------------ the same in 64 bits
def _pairs(x, H, rc):
    """All (i, j, d = x_j + n H - x_i) with |d| < rc in a periodic box."""
    n = x.shape[0]
    Hinv = torch.linalg.inv(H)
    widths = [1.0 / torch.linalg.norm(Hinv[:, a]).item() for a in range(3)]
    few = min(widths) > 2 * rc * (1 + 1e-9)
    if few:
        images = [(0, 0, 0)]
    else:
        m = [int(math.ceil(rc / w)) for w in widths]
        images = [(a, b, c) for a in range(-m[0], m[0] + 1) for b in range(-m[1], m[1] + 1) for c in range(-m[2], m[2] + 1)]
    s = x @ Hinv
    x = x - torch.floor(s) @ H
    got = []
    step = max(1, min(n, int(6e7 // n)))
    for b in range(0, n, step):
        base = x[None, :, :] - x[b:b + step, None, :]
        for im in images:
            if few:
                d = base - torch.round(base @ Hinv) @ H
            else:
                d = base + torch.tensor(im, dtype=x.dtype, device=x.device) @ H
            near = (d * d).sum(-1) < rc * rc
            if im == (0, 0, 0):
                k = torch.arange(near.shape[0], device=x.device)
                near[k, k + b] = False
            i, j = torch.nonzero(near, as_tuple=True)
            got.append((i + b, j, d[i, j]))
    i, j, d = (torch.cat([g[k] for g in got]) for k in range(3))
    order = torch.argsort(i, stable=True)
    return i[order], j[order], d[order]


class _Model:
    """The network of the library's header in plain torch, on the parameter vector theta."""

    def __init__(self, w, theta=None):
        t = torch.tensor(w.theta, dtype=torch.float64, device="cuda") if theta is None else theta
        self.w, self.p = w, {}
        for name, shape, off in synth.theta_layout(w.ntypes)[0]:
            self.p[name] = t[off:off + int(np.prod(shape))].reshape(shape)
        self.avg = torch.tensor(w.davg, device="cuda")
        self.std = torch.tensor(w.dstd, device="cuda")

    def net(self, ti, tj, s):
        p, n = self.p, f"emb{ti}{tj}."
        h1 = torch.tanh(s[:, None] * p[n + "W1"] + p[n + "b1"])
        h2 = torch.cat([h1, h1], 1) + torch.tanh(h1 @ p[n + "W2"] + p[n + "b2"])
        return torch.cat([h2, h2], 1) + torch.tanh(h2 @ p[n + "W3"] + p[n + "b3"])

    def rows(self, d, ti):
        """Normalised environment rows of pair vectors d of centres of type ti."""
        w = self.w
        r = torch.sqrt((d * d).sum(1))
        u = (r - w.rcut_smth) / (w.rcut - w.rcut_smth)
        if w.switch_kind:
            sw = 0.5 * torch.cos(math.pi * u) + 0.5
        else:
            sw = u ** 3 * (-6 * u * u + 15 * u - 10) + 1
        sw = torch.where(r < w.rcut_smth, torch.ones_like(r), sw)
        s = sw / r
        return (torch.cat([s[:, None], (s / r)[:, None] * d], 1) - self.avg[ti]) / self.std[ti]

    def energies(self, ti, n, rows):
        """E of n atoms of type ti; rows[tj] = (local atom, pair vectors)."""
        w, p = self.w, self.p
        T = torch.zeros(n, 400, dtype=torch.float64, device="cuda")
        for tj in range(w.ntypes):
            i, d = rows[tj]
            R = self.rows(d, ti)
            G = self.net(ti, tj, R[:, 0])
            T = T.index_add(0, i, (R[:, :, None] * G[:, None, :]).reshape(-1, 400))
            pad = (-self.avg[ti] / self.std[ti])
            free = w.sel[tj] - torch.bincount(i, minlength=n).to(torch.float64)
            T = T + free[:, None] * (pad[:, None] * self.net(ti, tj, pad[:1])).reshape(1, 400)
        T = T.reshape(n, 4, 100) / sum(w.sel)
        D = (T.transpose(1, 2) @ T[:, :, :16]).reshape(n, 1600)
        f = f"fit{ti}."
        h = torch.tanh(D @ p[f + "W1"] + p[f + "b1"])
        h = h + torch.tanh(h @ p[f + "W2"] + p[f + "b2"])
        h = h + torch.tanh(h @ p[f + "W3"] + p[f + "b3"])
        return (h @ p[f + "w4"].reshape(-1, 1)).reshape(-1) + p[f + "b4"] + p["e_bias"][ti]


def _chunks(types, i, atoms):
    """Chunks of one centre type: (ti, their atoms, the rows of i that belong to them)."""
    for ti in range(int(types.max()) + 1):
        of = torch.nonzero(types == ti).reshape(-1)
        for b in range(0, len(of), atoms):
            a = of[b:b + atoms]
            local = torch.full((len(types),), -1, dtype=torch.long, device="cuda")
            local[a] = torch.arange(len(a), device="cuda")
            r = torch.nonzero(local[i] >= 0).reshape(-1)
            yield ti, a, local, r


def _evaluate(model, x, types, H):
    i, j, d = _pairs(x, H, model.w.rcut)
    e = torch.zeros(len(types), dtype=torch.float64, device="cuda")
    g = torch.zeros_like(d)
    with torch.enable_grad():
        for ti, a, local, r in _chunks(types, i, 2048):
            dr = d[r].requires_grad_(True)
            rows = []
            for tj in range(model.w.ntypes):
                k = torch.nonzero(types[j[r]] == tj).reshape(-1)
                rows.append((local[i[r[k]]], dr[k]))
            ea = model.energies(ti, len(a), rows)
            (gr,) = torch.autograd.grad(ea.sum(), dr)
            e[a], g[r] = ea.detach(), gr
    F = torch.zeros_like(x).index_add(0, i, g).index_add(0, j, -g)
    return {"energy": e.sum().reshape(1), "atom_energy": e, "forces": F, "virial": -(g.T @ d)}


def _wrap(x, H):
    return x - torch.floor(x @ torch.linalg.inv(H)) @ H


def _md(model, x, v, types, H, mass, steps):
    x = _wrap(x, H)
    m = mass[types.long()][:, None]
    o = _evaluate(model, x, types, H)
    for k in range(steps):
        v = v + 0.5 * DT * KAPPA * o["forces"] / m
        x = x + DT * v
        if (k + 1) % EVERY == 0:
            x = _wrap(x, H)
        o = _evaluate(model, x, types, H)
        v = v + 0.5 * DT * KAPPA * o["forces"] / m
    ke = 0.5 * (m * v * v).sum() / KAPPA
    return {"x": x, "v": v, "forces": o["forces"], "potential": o["energy"], "kinetic": ke.reshape(1),
            "virial": o["virial"][None]}


def _train(w, h, prec):
    theta = torch.tensor(w.theta, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    theta = theta.to(torch.float64).requires_grad_(True)
    x = torch.tensor(h["x"], device="cuda")
    types = torch.tensor(h["types"], device="cuda")
    H = torch.tensor(h["boxes"][0].reshape(3, 3), device="cuda")
    base = _evaluate(_Model(w, theta.detach()), x, types, H)
    dF = base["forces"] - torch.tensor(h["F0"], device="cuda")
    dE = float(base["energy"]) - h["E0"]
    loss = h["cE"] * dE * dE + h["cF"] * (dF * dF).sum()
    # dL/dtheta = 2 cE dE dE/dtheta + sum 2 cF dF . dF/dtheta with F = -dE/dx, summed over chunks of centres
    wdir = 2 * h["cF"] * dF
    i, j, d = _pairs(x, H, w.rcut)
    grad = torch.zeros_like(theta)
    for ti, a, local, r in _chunks(types, i, 256):
        model = _Model(w, theta)
        dr = d[r].requires_grad_(True)
        rows = []
        for tj in range(w.ntypes):
            k = torch.nonzero(types[j[r]] == tj).reshape(-1)
            rows.append((local[i[r[k]]], dr[k]))
        e = model.energies(ti, len(a), rows).sum()
        (g,) = torch.autograd.grad(e, dr, create_graph=True)
        psi = 2 * h["cE"] * dE * e + (g * (wdir[i[r]] - wdir[j[r]])).sum()
        (gt,) = torch.autograd.grad(psi, theta)
        grad += gt
    return {"loss": loss.reshape(()), "grad": grad}


def exact(case, seed):
    n, rows = _rows(case)
    if rows * (case.get("steps", 0) + 1) > 1e8:
        return None  # over about 20 seconds
    h = _inputs(case, seed)
    w = _weights(case)
    if case["kind"] == "train":
        return _train(w, h, case["precision"])
    model = _Model(w)
    mass = torch.tensor(h["masses"], device="cuda")
    parts = []
    for k in range(len(h["offs"]) - 1):
        of = slice(int(h["offs"][k]), int(h["offs"][k + 1]))
        x = torch.tensor(h["x"][of], device="cuda")
        types = torch.tensor(h["types"][of], device="cuda")
        H = torch.tensor(h["boxes"][k].reshape(3, 3), device="cuda")
        if "steps" in case:
            parts.append(_md(model, x, torch.tensor(h["v"][of], device="cuda"), types, H, mass, case["steps"]))
        else:
            parts.append(_evaluate(model, x, types, H))
    if case["kind"] == "batch_compute":
        for p in parts:
            p["virial"] = p["virial"][None]
    return {q: torch.cat([p[q] for p in parts]) for q in parts[0]} if len(parts) > 1 else parts[0]
