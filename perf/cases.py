"""What is measured: the calls a user of this framework makes, at the sizes they are made at.

A case names a call of `paper_1909_11474_gb300.binding` (eval, fitness, param_grad, ga_step, md_force, md_nve), the
cells it works on and the sizes:

* cells "bulk": 64-atom diamond cells, strained by up to 2 % and displaced by 0.1 A (the GA training set); "mixed":
  supercells of 1 to 4 conventional cells per axis with up to two vacancies (7 to 512 atoms, strain 3 %, displacements
  of 0.05 to 0.2 A); "unit": the conventional 8-atom cell under small strains (elastic constants);
* C cells, P parameter sets ("population": genes uniform over +-30 % around the published parameters; "newton": a point
  near them and small steps along every parameter, what one iteration of the polish evaluates);
* precision 32 or 64, the minimal or the Tersoff form, and "rebuild": whether the pass rebuilds the neighbour lists (a new
  set of positions) or works on the build that the program keeps.

A call with precision 32 (and the gradient, which always works in it) computes in 32 bits and hands its sums out in 64-bit
buffers; `run` returns such values as the 32-bit numbers that they are accurate to. Calls with precision 64 return theirs
as they come. `exact` is the potential written out in plain torch in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1909_11474_gb300 import binding

R1, R2, MAX_NBR = 2.8, 3.2, 16
LATTICE = 5.431                                   # A, diamond Si
SI_MASS = 28.0855                                 # amu
ACCEL = 9.648533215665e-3                         # 1 eV/(A amu) in A/fs^2
KINETIC = 103.6426965268                          # 1 amu A^2/fs^2 in eV
# published minimal-Tersoff parameters (D0, alpha, r0, beta, n, h), and a set of the general form of like magnitude
MINIMAL = np.array([3.21481, 1.43134, 2.23801, 0.282818, 0.602568, -0.641048])
TERSOFF = np.array([3.2, 1.45, 2.25, 1.9, 0.65, -0.6, 0.06, 20.0, 3.0])   # D0, alpha, r0, S, n, h, gamma, c, d
# operations per atom of four bonds (50 a bond, 37 an ordered bond pair, 10 an atom), with the geometry in MD calls
FLOP_ATOM, FLOP_ATOM_MD = 654, 744


def listed():
    return [
        # one training cell under a handful of parameter sets, from its positions: the smallest call, tried first
        {"name": "single_cell", "call": "eval", "cells": "bulk", "C": 1, "P": 8, "precision": 32, "form": "minimal",
         "sets": "population", "rebuild": True},
        # the four strained 8-atom cells of the elastic constants, in FP64, from their positions
        {"name": "elastic_cells", "call": "eval", "cells": "unit", "C": 4, "P": 1, "precision": 64, "form": "minimal",
         "sets": "newton", "rebuild": True},
        # the genetic operators of one generation of the published population size
        {"name": "ga_step", "call": "ga_step", "P": 200, "G": 6},
        # one GA generation from scratch: new positions, lists, fitness of 200 sets on 300 cells (the headline workload)
        {"name": "ga_generation", "call": "fitness", "cells": "bulk", "C": 300, "P": 200, "precision": 32,
         "form": "minimal", "sets": "population", "rebuild": True},
        # the same generation's fitness in the nine-parameter form, on the lists that a fit keeps
        {"name": "fitness_tersoff", "call": "fitness", "cells": "bulk", "C": 300, "P": 200, "precision": 32,
         "form": "tersoff", "sets": "population", "rebuild": False},
        # a large population on a training set of ragged cells: the largest call
        {"name": "fitness_mixed", "call": "fitness", "cells": "mixed", "C": 500, "P": 1000, "precision": 32,
         "form": "minimal", "sets": "population", "rebuild": False},
        # one iteration of the finite-difference polish: 73 sets, FP64 fitness
        {"name": "fitness_fp64", "call": "fitness", "cells": "bulk", "C": 100, "P": 73, "precision": 64,
         "form": "minimal", "sets": "population", "rebuild": False},
        # predictions (energy, every force, virial) of a part of the population on the training set
        {"name": "eval_forces", "call": "eval", "cells": "bulk", "C": 300, "P": 64, "precision": 32, "form": "minimal",
         "sets": "population", "rebuild": False},
        # gradients of many candidates
        {"name": "gradient", "call": "grad", "cells": "bulk", "C": 100, "P": 64, "precision": 32, "form": "minimal",
         "sets": "population", "rebuild": False},
        # one iteration of the Newton polish (the point and two steps along each of six parameters) on ragged cells
        {"name": "polish_mixed", "call": "grad", "cells": "mixed", "C": 500, "P": 13, "precision": 32,
         "form": "minimal", "sets": "newton", "rebuild": False},
        # the force call of a 512,000-atom crystal
        {"name": "md_force", "call": "md_force", "n0": 40, "n1": 40, "n2": 40, "vacancies": 0, "sheared": False,
         "precision": 32},
        # twenty steps of molecular dynamics of 4,096 atoms at 300 K, in the integrator's default precision
        {"name": "md_nve", "call": "md_nve", "n0": 8, "n1": 8, "n2": 8, "vacancies": 0, "sheared": False,
         "precision": 64, "steps": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_ATOMS = {"bulk": 64, "mixed": 125, "unit": 8}


def draw(rng):
    call = rng.choice(["eval", "fitness", "fitness", "fitness", "grad", "grad", "md_force", "md_force", "md_nve", "ga_step"])
    if call == "ga_step":
        return {"call": call, "P": _log(rng, 20, 4096), "G": rng.choice([6, 6, 9])}
    if call in ("md_force", "md_nve"):
        nve = call == "md_nve"
        hi = 16 if nve else 40
        n = [_log(rng, 3, hi) for _ in range(3)]
        c = {"call": call, "n0": n[0], "n1": n[1], "n2": n[2], "vacancies": rng.randint(0, 9),
             "sheared": rng.random() < 0.3, "precision": rng.choice([64, 64, 32]) if nve else rng.choice([32, 32, 64])}
        if nve:
            c["steps"] = max(2, min(_log(rng, 2, 40), 400000 // (8 * n[0] * n[1] * n[2])))
        return c
    form = "tersoff" if call != "eval" and rng.random() < 0.2 else "minimal"
    precision = 64 if call != "grad" and rng.random() < 0.3 else 32
    cells = rng.choice(["bulk", "bulk", "mixed", "unit"] if precision == 64 else ["bulk", "bulk", "mixed"])
    C = _log(rng, 1, 500)
    low, high = {"eval": (1 if precision == 64 else 8, 200), "fitness": (20, 1000), "grad": (13, 200)}[call]
    P = _log(rng, low, high)
    # atom evaluations of a pass, so that none costs more than the largest listed case
    most = 6e5 if precision == 64 else {"eval": 1.5e7, "fitness": 5e7, "grad": 3e6}[call]
    C = min(C, int(most // (low * _ATOMS[cells])))
    P = min(P, int(most // (C * _ATOMS[cells])))
    return {"call": call, "cells": cells, "C": C, "P": P, "precision": precision, "form": form,
            "sets": "newton" if form == "minimal" and P < 20 else "population", "rebuild": rng.random() < 0.4}


# ---- inputs -------------------------------------------------------------------------------------------------------

_BASIS = np.concatenate([np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]]),
                         np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]]) + 0.25])


def _diamond(reps, a=LATTICE):
    g = np.stack(np.meshgrid(*(np.arange(m) for m in reps), indexing="ij"), -1).reshape(-1, 1, 3)
    return (g + _BASIS[None]).reshape(-1, 3) * a, np.diag(np.asarray(reps, dtype=np.float64) * a)


def _strain(rng, s):
    e = rng.uniform(-s, s, 6)
    return np.eye(3) + np.array([[e[0], e[3], e[5]], [e[3], e[1], e[4]], [e[5], e[4], e[2]]])


def _cells(case, rng):
    """Positions [N][3], boxes [C][3][3] and atom offsets [C + 1] of the case's cells."""
    pos, box = [], []
    for _ in range(case["C"]):
        kind = case["cells"]
        if kind == "bulk":
            x, H = _diamond((2, 2, 2))
            m, sigma, vac = _strain(rng, 0.02), 0.1, 0
        elif kind == "mixed":
            x, H = _diamond(rng.integers(1, 5, 3))
            m, sigma, vac = _strain(rng, 0.03), rng.uniform(0.05, 0.2), int(rng.integers(0, 3))
        else:
            x, H = _diamond((1, 1, 1), rng.uniform(5.40, 5.46))
            m, sigma, vac = _strain(rng, 1e-3), 0.02, 0
        if vac:
            x = x[np.sort(rng.choice(len(x), len(x) - vac, replace=False))]
        pos.append(x @ m.T + rng.normal(0.0, sigma, x.shape))
        box.append(H @ m.T)
    off = np.concatenate([[0], np.cumsum([len(x) for x in pos])]).astype(np.int32)
    return np.ascontiguousarray(np.concatenate(pos)), np.ascontiguousarray(np.stack(box)), off


def _sets(case, rng):
    P = case["P"]
    if case["form"] == "tersoff":
        return TERSOFF * rng.uniform(0.95, 1.05, (P, 9))
    if case["sets"] == "newton":                   # the point, then steps of 1e-4 of the +-30 % range, along each parameter
        x = np.tile(MINIMAL * rng.uniform(0.98, 1.02, 6), (P, 1))
        for k in range(1, P):
            x[k, (k - 1) % 6] += (1e-4 if k <= 6 else -1e-4) * 0.6 * abs(MINIMAL[(k - 1) % 6])
        return x
    return MINIMAL + 0.3 * np.abs(MINIMAL) * rng.uniform(-1.0, 1.0, (P, 6))


def _crystal(case, rng):
    x, H = _diamond((case["n0"], case["n1"], case["n2"]))
    if case["vacancies"]:
        x = np.delete(x, rng.choice(len(x), case["vacancies"], replace=False), axis=0)
    if case["sheared"]:
        m = _strain(rng, 0.02)
        x, H = x @ m.T, H @ m.T
    return np.ascontiguousarray(x + rng.normal(0.0, 0.08 if case["call"] == "md_force" else 0.02, x.shape)), H


def _dynamics(case, seed):
    """A crystal at 300 K: positions, box, masses, velocities."""
    rng = np.random.default_rng(seed)
    pos, H = _crystal(case, rng)
    mass = np.full(len(pos), SI_MASS)
    vel = rng.normal(0.0, math.sqrt(8.617333262e-5 * 300.0 / SI_MASS * ACCEL), pos.shape)
    return pos, H, mass, vel - vel.mean(0)


def _genes(case, seed):
    rng = np.random.default_rng(seed)
    P, G = case["P"], case["G"]
    centre = MINIMAL if G == 6 else TERSOFF
    lo, hi = centre - 0.3 * np.abs(centre), centre + 0.3 * np.abs(centre)
    Z = np.exp(rng.normal(0.0, 1.0, P))
    Z[rng.random(P) < 0.02] = math.inf             # sets whose prediction was not finite
    n_par = P // 2
    u = rng.random((G + 2) * (P - n_par) + 2 * G * (P - 1))
    return Z, rng.random((P, G)), u, lo, hi, n_par, 0.1


def _training(case, seed, dev):
    """Cells, parameter sets and targets: the published potential's predictions and noise, as training data have it."""
    rng = np.random.default_rng(seed)
    pos, box, off = _cells(case, rng)
    x = _sets(case, rng)
    tg = None
    if case["call"] != "eval":
        g = _geometry(pos, box, off, dev)
        E, F, W = _evaluate(g, torch.tensor(MINIMAL[None], device=dev))
        nat = np.diff(off).astype(np.float64)
        tg = {"E": E[0].cpu().numpy() / nat + rng.normal(0.0, 1e-3, len(nat)),
              "W": W[0].cpu().numpy() / nat[:, None] + rng.normal(0.0, 5e-3, (len(nat), 6)),
              "F": F[0].cpu().numpy() + rng.normal(0.0, 0.02, pos.shape),
              "mask": np.full(len(nat), 7, np.uint8)}
    return pos, box, off, x, tg


def prepare(case, seed):
    dev = torch.device("cuda")
    put = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
    s = {"case": case}
    if case["call"] == "ga_step":
        Z, genes, u, lo, hi, n_par, rate = _genes(case, seed)
        s.update(Z=put(Z), genes=put(genes), u=put(u), lo=put(lo), hi=put(hi), n_par=n_par, rate=rate,
                 genes_out=torch.empty_like(put(genes)), params=torch.empty_like(put(genes)),
                 order=torch.empty(len(Z), dtype=torch.int32, device=dev))
        return s
    s["ctx"] = binding.Context(0)
    if case["call"] == "md_force":
        pos, H = _crystal(case, np.random.default_rng(seed))
        s.update(pos=put(pos), box=H)
        return s
    if case["call"] == "md_nve":
        pos, H, mass, vel = _dynamics(case, seed)
        s.update(pos=put(pos), box=H, mass=put(mass), vel=put(vel))
        return s
    pos, box, off, x, tg = _training(case, seed, dev)
    s.update(pos=put(pos), box=put(box), off=off, params=put(x))
    if tg is not None:
        s["targets"] = {k: put(v) for k, v in tg.items()}
        s["Z"] = torch.empty(case["P"], dtype=torch.float64, device=dev)
    if case["form"] == "tersoff":
        s["ctx"].set_form(binding.FORM_TERSOFF)
    if not case["rebuild"]:
        s["ctx"].build_neighbors(off, s["pos"], s["box"], R1, R2, MAX_NBR)
    return s


def run(state):
    s, c = state, state["case"]
    call, ctx = c["call"], state.get("ctx")
    if call == "ga_step":
        binding.ga_step(s["Z"], s["genes"], s["u"], s["lo"], s["hi"], s["n_par"], s["rate"], s["genes_out"], s["params"],
                        s["order"])
        return {"genes": s["genes_out"], "params": s["params"], "order": s["order"]}
    as32 = (lambda t: t.float()) if c["precision"] == 32 else (lambda t: t)
    if call == "md_force":
        E, F, W = ctx.md_force(s["pos"], s["box"], MINIMAL, R1, R2, MAX_NBR, precision=c["precision"])
        return {"E": as32(E), "F": F, "W": as32(W)}
    if call == "md_nve":                           # a further stretch of the trajectory: pos and vel move on
        Ep, Ek, F, W = ctx.md_nve(s["pos"], s["vel"], s["mass"], s["box"], MINIMAL, 1.0, c["steps"], R1, R2, MAX_NBR,
                                  precision=c["precision"])
        return {"pos": s["pos"], "vel": as32(s["vel"]), "Epot": as32(Ep), "Ekin": as32(Ek), "F": F, "W": as32(W)}
    if c["rebuild"]:
        ctx.build_neighbors(s["off"], s["pos"], s["box"], R1, R2, MAX_NBR)
    if call == "eval":
        E, F, W = ctx.eval(s["params"], precision=c["precision"])
        return {"E": as32(E), "F": F, "W": as32(W)}
    if call == "fitness":
        Z, _, _ = ctx.fitness(s["params"], s["targets"], precision=c["precision"], out=(s["Z"], None, None))
        return {"Z": as32(Z)}
    L, dL = ctx.param_grad(s["params"], s["targets"])
    return {"L": as32(L), "dL": as32(dL)}


def work(case):
    call = case["call"]
    if call == "ga_step":
        P, G = case["P"], case["G"]
        n_u = (G + 2) * (P - P // 2) + 2 * G * (P - 1)
        return {"bytes": 8 * (P + 3 * P * G + n_u + 2 * G) + 4 * P, "flops": P * (math.log2(P) + 3 * G)}
    if call in ("md_force", "md_nve"):
        N = 8 * case["n0"] * case["n1"] * case["n2"] - case["vacancies"]
        fb = 12 if case["precision"] == 32 else 24
        if call == "md_force":
            return {"bytes": N * (24 + fb), "flops": N * FLOP_ATOM_MD}
        steps = case["steps"]                      # each step: positions and velocities read and written
        return {"bytes": N * (96 * steps + fb + 8), "flops": N * (FLOP_ATOM_MD * (steps + 1) + 24 * steps)}
    C, P = case["C"], case["P"]
    N = C * _ATOMS[case["cells"]]
    nx = 9 if case["form"] == "tersoff" else 6
    flop = FLOP_ATOM + (12 * 6 if case["form"] == "tersoff" else 0)
    inputs = 24 * N + 72 * C + 8 * nx * P
    if call == "eval":
        return {"bytes": inputs + P * (56 * C + (12 if case["precision"] == 32 else 24) * N), "flops": P * N * flop}
    inputs += 24 * N + 57 * C
    if call == "fitness":
        return {"bytes": inputs + 8 * P, "flops": P * N * flop}
    return {"bytes": inputs + 8 * P * (1 + nx), "flops": 3 * P * N * flop}    # values and a reverse sweep


# ---- the potential in plain torch, 64 bits -------------------------------------------------------------------------

def _dot(n, H):
    """n . H for integer image indices n [..., 3] and box rows H [3][3], component by component."""
    return torch.stack([n[..., 0] * H[0, k] + n[..., 1] * H[1, k] + n[..., 2] * H[2, k] for k in range(3)], -1)


def _bonds(x, H):
    """Owner, partner, vector and image of every bond of a small cell (each plane spacing above two thirds of R2)."""
    s = _dot(x, torch.linalg.inv(H.cpu()).to(x.device))
    base = -torch.round(s[None, :, :] - s[:, None, :])                     # [i][j]
    offs = torch.tensor([[a, b, c] for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)], dtype=x.dtype,
                        device=x.device)
    n = base[None] + offs[:, None, None, :]
    d = (x[None, :, :] - x[:, None, :])[None] + _dot(n, H)
    hit = (d * d).sum(-1) < R2 * R2
    same = torch.eye(len(x), dtype=torch.bool, device=x.device)[None] & (n == 0).all(-1)
    o, i, j = torch.nonzero(hit & ~same, as_tuple=True)
    return i, j, d[o, i, j], n[o, i, j].long()


def _bonds_large(x, H):
    """The same for a large cell, by a cell list (at least three cells along each axis)."""
    Hi = torch.linalg.inv(H.cpu()).to(x.device)
    nc = torch.floor(1.0 / (Hi.norm(dim=0) * R2)).long()                   # plane spacing k = 1 / |column k of H^-1|
    w = torch.floor(_dot(x, Hi) * nc).long()
    m = torch.div(w, nc, rounding_mode="floor")
    c = w - m * nc
    flat = lambda v: (v[:, 0] * nc[1] + v[:, 1]) * nc[2] + v[:, 2]  # noqa: E731
    cell = flat(c)
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=int(nc.prod()))
    start = torch.cumsum(count, 0) - count
    cap = int(count.max())
    table = torch.full((len(count), cap), -1, dtype=torch.long, device=x.device)
    table[cell[order], torch.arange(len(x), device=x.device) - start[cell[order]]] = order
    out = []
    for o in [(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)]:
        v = c + torch.tensor(o, device=x.device)
        k = torch.div(v, nc, rounding_mode="floor")
        j = table[flat(v - k * nc)]                                          # [N][cap]
        n = k[:, None, :] + m[:, None, :] - m[j.clamp(min=0)]
        d = x[j.clamp(min=0)] - x[:, None, :] + _dot(n.to(x.dtype), H)
        own = torch.arange(len(x), device=x.device)[:, None]
        hit = (j >= 0) & ((d * d).sum(-1) < R2 * R2) & ~((j == own) & (n == 0).all(-1))
        i, t = torch.nonzero(hit, as_tuple=True)
        out.append((i, j[i, t], d[i, t], n[i, t]))
    return tuple(torch.cat(p) for p in zip(*out))


def _geometry(pos, box, off, dev):
    """Padded bond arrays [atoms][M] of all cells: vectors, which are there, and each bond's reverse."""
    x, boxes = torch.tensor(pos, device=dev), torch.tensor(box, device=dev)
    parts = []
    for c in range(len(off) - 1):
        a, b = int(off[c]), int(off[c + 1])
        i, j, d, n = (_bonds if b - a <= 1024 else _bonds_large)(x[a:b], boxes[c])
        parts.append((i + a, j + a, d, n))
    return _padded(*(torch.cat(p) for p in zip(*parts)), len(x), np.asarray(off), dev)


def _padded(i, j, d, n, N, off, dev):
    by = torch.argsort(i, stable=True)
    i, j, d, n = i[by], j[by], d[by], n[by]
    count = torch.bincount(i, minlength=N)
    M = max(1, int(count.max()))
    slot = i * M + torch.arange(len(i), device=dev) - (torch.cumsum(count, 0) - count)[i]
    code = lambda v: ((v[:, 0] + 512) * 1024 + v[:, 1] + 512) * 1024 + v[:, 2] + 512  # noqa: E731
    pair = i * N + j                                # bonds sorted by (pair, image), looked up by (reverse pair, -image)
    images, at = torch.unique(torch.cat([code(n), code(-n)]), return_inverse=True)
    fwd = pair * len(images) + at[: len(i)]
    rev = (j * N + i) * len(images) + at[len(i):]
    srt = torch.argsort(fwd)
    back = slot[srt[torch.searchsorted(fwd[srt], rev)]]
    vec = torch.zeros((N * M, 3), dtype=torch.float64, device=dev)
    vec[:, 0] = 1.0
    vec[slot] = d
    there = torch.zeros(N * M, dtype=torch.float64, device=dev)
    there[slot] = 1.0
    reverse = torch.zeros(N * M, dtype=torch.long, device=dev)
    reverse[slot] = back
    nat = np.diff(off)
    idx = np.minimum(off[:-1, None] + np.arange(nat.max())[None], off[1:, None] - 1)   # atoms of every cell, padded
    inside = np.arange(nat.max())[None] < nat[:, None]
    return {"d": vec.view(N, M, 3), "there": there.view(N, M), "rev": reverse,
            "atoms": torch.tensor(idx, dtype=torch.long, device=dev),
            "inside": torch.tensor(inside, dtype=torch.float64, device=dev), "nat": torch.tensor(nat, device=dev)}


def _evaluate(g, x):
    """E [P][C], F [P][N][3] and W [P][C][6] of the parameter sets x [P][6 or 9]."""
    d, there = g["d"], g["there"]
    N, M, _ = d.shape
    r = d.norm(dim=-1)
    u = d / r[..., None]
    w = (r - R1) / (R2 - R1)
    mid = (r > R1) & (r < R2)
    fc = there * torch.where(mid, 0.5 * (1.0 + torch.cos(math.pi * w)), torch.where(r <= R1, 1.0, 0.0))
    fcp = there * torch.where(mid, -0.5 * math.pi / (R2 - R1) * torch.sin(math.pi * w), 0.0)
    cos = torch.einsum("njk,nlk->njl", u, u)
    pairs = there[:, :, None] * there[:, None, :] * (1.0 - torch.eye(M, dtype=d.dtype, device=d.device))
    p = [x[:, k][:, None, None] for k in range(x.shape[1])]
    if x.shape[1] == 6:
        D0, al, r0, beta, n, h = p
        S = 2.0
    else:
        D0, al, r0, S, n, h, gamma, c, dd = p
    lam, mu = al * (2.0 * S) ** 0.5, al * (2.0 / S) ** 0.5
    fR = D0 / (S - 1.0) * torch.exp(-lam * (r - r0))
    fA = D0 * S / (S - 1.0) * torch.exp(-mu * (r - r0))
    v = cos - h[..., None]                                                   # [P][N][M][M]
    if x.shape[1] == 6:
        gg, gp = beta[..., None] * v * v, 2.0 * beta[..., None] * v
    else:
        c2, d2, ga = (c * c)[..., None], (dd * dd)[..., None], gamma[..., None]
        gg, gp = ga * c2 / d2 * v * v / (d2 + v * v) + ga, 2.0 * ga * c2 * v / (d2 + v * v) ** 2
    zeta = (pairs * fc[:, None, :] * gg).sum(-1).clamp(min=1e-30)
    zn = zeta ** n
    b = (1.0 + zn) ** (-0.5 / n)
    bp = -0.5 * b * zn / (zeta * (1.0 + zn))
    cc = -0.5 * fc * fA * bp
    rad = 0.5 * (fcp * (fR - b * fA) + fc * (-lam * fR + mu * b * fA))
    wt = pairs * (cc[..., :, None] * fc[:, None, :] + cc[..., None, :] * fc[:, :, None]) * gp
    A = torch.einsum("pnjl,nlk->pnjk", wt, u)
    coef = rad - (wt * cos).sum(-1) / r + fcp * (pairs * cc[..., None, :] * gg).sum(-1)
    Pij = there[..., None] * (coef[..., None] * u + A / r[..., None])        # dU_i/dd_ij
    Ui = 0.5 * (fc * (fR - b * fA)).sum(-1)
    back = Pij.reshape(len(x), N * M, 3)[:, g["rev"]].reshape(Pij.shape) * there[..., None]
    F = (Pij - back).sum(2)
    V = -torch.einsum("nja,pnjb->pnab", d * there[..., None], Pij)
    Wi = torch.stack([V[..., 0, 0], V[..., 1, 1], V[..., 2, 2], V[..., 0, 1], V[..., 1, 2], V[..., 2, 0]], -1)
    E = (Ui[:, g["atoms"]] * g["inside"]).sum(-1)
    W = (Wi[:, g["atoms"]] * g["inside"][..., None]).sum(2)
    return E, F, W


def _residuals(g, x, tg):
    """S [P][3] and D [3] of the fitness."""
    E, F, W = _evaluate(g, x)
    nat = g["nat"].double()
    S = torch.stack([((E / nat - tg["E"]) ** 2).sum(-1), ((W / nat[:, None] - tg["W"]) ** 2).sum((-1, -2)),
                     ((F - tg["F"]) ** 2).sum((-1, -2))], -1)
    return S, torch.stack([(tg[k] ** 2).sum() for k in ("E", "W", "F")])


def _exact_genes(case, seed):
    Z, genes, u, lo, hi, n_par, rate = _genes(case, seed)
    P, G = genes.shape
    order = np.argsort(np.where(np.isfinite(Z), Z, np.inf), kind="stable")
    new = genes[order].copy()
    kid = u[: (G + 2) * (P - n_par)].reshape(P - n_par, G + 2)
    pa, pb = (np.minimum((kid[:, k] * n_par).astype(int), n_par - 1) for k in (0, 1))
    new[n_par:] = np.where(kid[:, 2:] < 0.5, genes[order[pa]], genes[order[pb]])
    mut = u[(G + 2) * (P - n_par):].reshape(P - 1, G, 2)
    new[1:] = np.where(mut[..., 0] < rate, mut[..., 1], new[1:])
    return {"genes": torch.tensor(new), "params": torch.tensor(lo + new * (hi - lo)),
            "order": torch.tensor(order.astype(np.int32))}


def _one_cell(x, H):
    i, j, d, n = (_bonds if len(x) <= 512 else _bonds_large)(x, H)
    return _padded(i, j, d, n, len(x), np.array([0, len(x)]), x.device)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    call = case["call"]
    if call == "ga_step":
        return _exact_genes(case, seed)
    one = torch.tensor(MINIMAL[None], device=dev)
    if call == "md_force":
        pos, H = _crystal(case, np.random.default_rng(seed))
        E, F, W = _evaluate(_one_cell(torch.tensor(pos, device=dev), torch.tensor(H, device=dev)), one)
        return {"E": E[0], "F": F[0], "W": W[0, 0]}
    if call == "md_nve":
        pos, H, mass, vel = (torch.tensor(v, device=dev) for v in _dynamics(case, seed))
        kin = lambda v: 0.5 * KINETIC * (mass * (v * v).sum(-1)).sum()  # noqa: E731
        force = lambda x: _evaluate(_one_cell(x, H), one)  # noqa: E731
        acc = ACCEL / mass[:, None]
        E, F, W = force(pos)
        Ep, Ek = [E[0, 0]], [kin(vel)]
        for _ in range(case["steps"]):             # velocity Verlet, dt = 1 fs
            vel = vel + 0.5 * acc * F[0]
            pos = pos + vel
            E, F, W = force(pos)
            vel = vel + 0.5 * acc * F[0]
            Ep.append(E[0, 0])
            Ek.append(kin(vel))
        return {"pos": pos, "vel": vel, "Epot": torch.stack(Ep), "Ekin": torch.stack(Ek), "F": F[0], "W": W[0, 0]}
    pos, box, off, x, tg = _training(case, seed, dev)
    g, x = _geometry(pos, box, off, dev), torch.tensor(x, device=dev)
    if tg is not None:
        tg = {k: torch.tensor(v, device=dev) for k, v in tg.items()}
    N, M, _ = g["d"].shape
    step = max(1, int((1e8 if call == "grad" else 4e8) // (8 * N * M * M)))   # sets at a time
    got = []
    for k in range(0, len(x), step):
        xk = x[k: k + step].clone().requires_grad_(call == "grad")
        if call == "eval":
            got.append(_evaluate(g, xk))
            continue
        S, D = _residuals(g, xk, tg)
        if call == "fitness":
            got.append((torch.sqrt(S / D).sum(-1),))
        else:
            L = (S / D).sum(-1)
            got.append((L.detach(), torch.autograd.grad(L.sum(), xk)[0]))
    got = [torch.cat(v) for v in zip(*got)]
    return dict(zip({"eval": ("E", "F", "W"), "fitness": ("Z",), "grad": ("L", "dL")}[call], got))
