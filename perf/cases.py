"""Performance cases: what a user of this library has it do, through its public entry points.

  md          one time step of molecular dynamics with extrapolation control: the neighbor list is
              rebuilt for the moved atoms, then energies, forces, virial and (option) the grade of
              every neighborhood.  Crystals, alloys and a liquid, from a cell that a laptop holds to
              a million atoms; single ("mixed") and double precision.
  train       the loss and its gradient for a training set (the step of a fit), on the list built once.
  energy_grad energies of a batch with reverse-mode derivatives in positions and parameters
              (the torch.autograd wrapper: forward and backward).
  active_set  loading an active set: A^-1 of the m x m matrix.
  select      choosing an active set: parameter rows of a pool, then MaxVol over them.
  cut         what follows a flagged atom: its neighborhood and its spherical cluster.

A mixed-precision program keeps single-precision state, so the outputs of the mixed path (which the
library hands over in double containers) are taken as float32; the FP64 path's as they are.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2304_13144_gb300 import api, autograd, synth

# the configuration families of the workload table: (basis, lattice constant, displacement)
LATTICES = {
    "fcc": (np.array([[0, 0, 0], [0.5, 0.5, 0], [0.5, 0, 0.5], [0, 0.5, 0.5]]), 3.6, 0.1),
    "bcc": (np.array([[0, 0, 0], [0.5, 0.5, 0.5]]), 2.87, 0.08),
}
NBAR = {"fcc": 42.0, "bcc": 58.0, "liquid": 76.0, "train": 42.0}   # mean neighbor counts (parameter scale)
N_Q, R_MIN = 8, 2.0


# ------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------

def _md(name, lattice, nx, ny, nz, types, level, prec="mixed", grade=True, vacancies=0, r_cut=5.0):
    return {"name": name, "kind": "md", "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "types": types,
            "level": level, "prec": prec, "grade": grade, "vacancies": vacancies, "r_cut": r_cut}


def listed():
    return [
        # the smallest periodic cell in use: launches and round trips to the host
        _md("md_fcc_108_l8", "fcc", 3, 3, 3, 1, 8),
        # an ordinary MD cell of a ternary alloy, a vacancy in it
        _md("md_fcc_4k_l20", "fcc", 10, 10, 10, 3, 20, vacancies=1),
        # plain MD (no grade) of an ordered binary crystal
        _md("md_b2_128k_l16", "bcc", 40, 40, 40, 2, 16, grade=False),
        # the benchmark: MD with a grade per atom, a million atoms
        _md("md_fcc_1m_l20", "fcc", 64, 64, 64, 3, 20),
        # large neighborhoods: a quaternary liquid at the largest level
        _md("md_liquid_131k_l24", "liquid", 4, 4, 8, 4, 24, r_cut=6.0),
        # the same step all in double precision (reference runs, relaxations)
        _md("md_fcc_16k_l20_fp64", "fcc", 16, 16, 16, 3, 20, prec="fp64"),
        # one step of a fit, in the default precision of the fit and in the mixed one
        {"name": "train_512_l16_fp64", "kind": "train", "n_cfg": 512, "hi": 256, "types": 3, "level": 16,
         "prec": "fp64", "stress": False},
        {"name": "train_512_l16_mixed", "kind": "train", "n_cfg": 512, "hi": 256, "types": 3, "level": 16,
         "prec": "mixed", "stress": True},
        # the potential inside a differentiable program: a batch of small cells
        {"name": "energy_grad_64_l16", "kind": "energy_grad", "n_cfg": 64, "hi": 128, "types": 2, "level": 16,
         "prec": "fp64"},
        # an active set is loaded when a run starts and after every retraining
        {"name": "active_set_l20", "kind": "active_set", "types": 3, "level": 20, "n_q": 8},
        # active learning: candidates of a snapshot into the active set
        {"name": "select_2000_l16", "kind": "select", "nx": 10, "ny": 10, "nz": 10, "types": 2, "level": 16},
        # extrapolative atoms of a run are cut out for labelling
        {"name": "cut_32_of_16k", "kind": "cut", "nx": 20, "ny": 20, "nz": 20, "centers": 32, "radius": 8.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, per_cell):
    """Unequal cell counts for a log-uniform number of atoms in about [lo, hi]."""
    n = _log(rng, lo, hi)
    side = (n / per_cell) ** (1.0 / 3.0)
    nx = max(2, round(side * rng.uniform(0.8, 1.2)))
    ny = max(2, round(side * rng.uniform(0.8, 1.2)))
    nz = max(2, int(n / per_cell / (nx * ny)))
    return nx, ny, nz


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md", "train", "train", "energy_grad", "active_set", "select", "cut"])
    if kind == "md":
        lattice = rng.choice(["fcc", "fcc", "bcc", "liquid"])
        if lattice == "liquid":
            c = _md("", "liquid", rng.randint(1, 4), rng.randint(1, 4), rng.randint(1, 8), 4, 24,
                    grade=rng.random() < 0.5, r_cut=6.0)
        else:
            prec = "fp64" if rng.random() < 0.3 else "mixed"
            level = rng.choice([8, 12, 16, 20])
            nx, ny, nz = _box(rng, 100, 15000 if prec == "fp64" else 700000, 4 if lattice == "fcc" else 2)
            c = _md("", lattice, nx, ny, nz, rng.randint(1, 3), level, prec, rng.random() < 0.7)
        c["vacancies"] = rng.randint(1, 31)
        del c["name"]
        return c
    if kind in ("train", "energy_grad"):
        big = kind == "train"
        c = {"kind": kind, "n_cfg": _log(rng, 4, 500 if big else 64), "hi": rng.randint(16, 250 if big else 128),
             "types": rng.randint(1, 3), "level": rng.choice([8, 12, 16]),
             "prec": "mixed" if rng.random() < 0.4 else "fp64"}
        if big:
            c["stress"] = rng.random() < 0.5
        return c
    if kind == "active_set":
        types = rng.randint(1, 3)
        return {"kind": kind, "types": types, "level": rng.choice([8, 10, 12, 14, 16, 18, 20]), "n_q": rng.randint(5, 9)}
    if kind == "select":
        nx, ny, nz = _box(rng, 700, 2000, 2)
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "types": rng.randint(1, 2), "level": rng.choice([8, 12, 16])}
    nx, ny, nz = _box(rng, 250, 16000, 2)
    return {"kind": "cut", "nx": nx, "ny": ny, "nz": nz, "centers": _log(rng, 1, 100),
            "radius": round(rng.uniform(5.0, 8.0), 2)}


# ------------------------------------------------------------------------------------
# inputs (from the seed alone)
# ------------------------------------------------------------------------------------

def _rsa_cube(g, n, density=0.085, d_min=1.8):
    """n points in a periodic cube, added one batch at a time at least d_min from all others."""
    L = (n / density) ** (1.0 / 3.0)
    pos = np.empty((0, 3))

    def far(x, y):
        d = x[:, None, :] - y[None, :, :]
        d -= L * np.round(d / L)
        return (d * d).sum(-1) >= d_min * d_min

    while len(pos) < n:
        x = g.uniform(0.0, L, (256, 3))
        x = x[far(x, pos).all(1)]
        ok = far(x, x) | np.triu(np.ones((len(x), len(x)), bool))   # against earlier candidates
        pos = np.concatenate([pos, x[ok.all(1)]])[:n]
    return pos, L


def _crystal(case, seed, types):
    """One periodic configuration of the case's structure, `vacancies` atoms taken out."""
    g = synth.rng(seed)
    reps = (case["nx"], case["ny"], case["nz"])
    if case.get("lattice") == "liquid":
        cube, L = _rsa_cube(g, 1024)
        t = np.stack(np.meshgrid(*(np.arange(k) for k in reps), indexing="ij"), -1).reshape(-1, 3)
        pos = (cube[None] + L * t[:, None]).reshape(-1, 3)
        cell = np.diag([L * k for k in reps])
        species = g.integers(0, types, len(pos))
    else:
        basis, a, sigma = LATTICES[case.get("lattice", "bcc")]
        pos, cell, sub = synth.cubic_supercell(basis, a, reps)
        if len(basis) == 2 and types == 2:      # ordered, a tenth of the atoms on the other sublattice
            species = np.where(g.random(len(pos)) < 0.1, 1 - sub, sub)
        else:                                   # random solid solution of equal shares
            species = g.permutation(np.arange(len(pos)) % types)
        pos = pos + g.normal(0.0, sigma, pos.shape)
    gone = g.choice(len(pos), case.get("vacancies", 0), replace=False)
    return synth.single(np.delete(pos, gone, 0), np.delete(species, gone), cell)


def _theta(case, seed, nbar):
    """Parameters at the scale of the workload table."""
    basis = _basis(case["level"])
    return synth.draw_theta(seed, case["types"], _n_rad(case["level"]), case.get("n_q", N_Q),
                            [sum(nu for _, nu in labs) for labs, _ in basis], [len(labs) for labs, _ in basis],
                            R_MIN, case.get("r_cut", 5.0), nbar)


def _inputs(case, seed):
    """Host arrays of a case: batch, theta, and what else its kind takes."""
    kind, types = case["kind"], case.get("types", 2)
    x = {}
    if kind in ("train", "energy_grad"):
        # one set of cells per case; the seed moves the atoms and deals the species
        x["batch"] = b = synth.training_batch(3, case["n_cfg"], types, 8, case["hi"])
        x["theta"] = _theta(case, seed + 1, NBAR["train"])
        g = synth.rng(seed + 2)
        n, k = len(b["type"]), case["n_cfg"]
        b["pos"] = b["pos"] + g.normal(0.0, 0.05, (n, 3))
        b["type"] = g.integers(0, types, n).astype(np.int32)
        x["E_ref"] = g.normal(0.0, 0.1, k) * np.diff(b["atom_offset"])
        x["F_ref"] = g.normal(0.0, 0.5, (n, 3))
        x["W_ref"] = g.normal(0.0, 1.0, (k, 9))
        x["gE"] = g.normal(0.0, 1.0, k)
        return x
    if kind != "cut":
        x["theta"] = _theta(case, seed + 1, NBAR[case.get("lattice", "bcc")])
    m = len(x["theta"]) if "theta" in x else 0
    if kind == "active_set" or case.get("grade"):
        x["A"] = synth.diag_dominant(seed + 2, m)
    if kind != "active_set":
        x["batch"] = _crystal(case, seed, types)
        n = len(x["batch"]["type"])
        if kind == "select":
            n_rad = _n_rad(case["level"])
            x["pick"] = synth.sample_atoms(seed + 3, n, m - n_rad * (n_rad + 1) // 2)
        if kind == "cut":
            x["centers"] = synth.sample_atoms(seed + 3, n, min(n, case["centers"]))
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    s = {"case": case, "kind": case["kind"]}
    level = case.get("level", 8)
    desc = api.make_desc(case.get("types", 2), level, case.get("n_q", N_Q), R_MIN, case.get("r_cut", 5.0))
    if "batch" in x:
        s["batch"] = b = api.Batch(x["batch"])
    theta = x["theta"] if "theta" in x else np.zeros(api.mtp_describe(desc)["n_params"])
    s["model"] = model = api.mtp_load(desc, theta)
    if case["kind"] == "md":
        s["nbr"] = api.Neighbors()
        n, k = b.n_atoms, b.n_cfg
        dev = {"dtype": torch.float64, "device": "cuda"}
        s["out"] = out = {"energy": torch.empty(k, **dev), "site_energy": torch.empty(n, **dev),
                          "forces": torch.empty((n, 3), **dev), "virial": torch.empty((k, 3, 3), **dev)}
        if case["grade"]:
            api.mtp_set_active_set(model, torch.as_tensor(x["A"], device="cuda"))
            out["gamma"] = torch.empty(n, **dev)
            if case["prec"] == "fp64":
                out["argmax"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif case["kind"] == "energy_grad":
        s["pos"] = b.pos.clone().requires_grad_(True)
        s["theta"] = torch.tensor(theta, requires_grad=True)
        s["gE"] = torch.as_tensor(x["gE"], device="cuda")
    elif case["kind"] == "active_set":
        s["A"] = torch.as_tensor(x["A"], device="cuda")
    else:
        s["nbr"] = api.mtp_build_neighbors(model, b)
        if case["kind"] == "train":
            for k in ("E_ref", "F_ref", "W_ref"):
                s[k] = torch.as_tensor(x[k], device="cuda")
        elif case["kind"] == "select":
            s["pick"] = torch.as_tensor(x["pick"], device="cuda")
            D = torch.as_tensor(api.mtp_gauge_directions(desc, theta), device="cuda")
            s["gauge"] = D / D.norm(dim=1, keepdim=True)
        else:
            s["centers"] = torch.as_tensor(x["centers"], device="cuda")
    return s


def run(s):
    case, kind, model = s["case"], s["kind"], s["model"]
    if kind == "md":
        nbr = api.mtp_build_neighbors(model, s["batch"], s["nbr"])
        out = api.mtp_step(model, s["batch"], nbr, case["prec"], threshold=2.0, out=s["out"], grade=case["grade"])
        return out if case["prec"] == "fp64" else {k: v.float() for k, v in out.items()}
    if kind == "train":
        loss, grad = api.mtp_train_step(model, s["batch"], s["nbr"], s["E_ref"], s["F_ref"], s["W_ref"], 1.0, 0.01,
                                        1e-3 if case["stress"] else 0.0, case["prec"])
        return [loss, grad] if case["prec"] == "fp64" else [loss.float(), grad.float()]
    if kind == "energy_grad":
        s["pos"].grad = s["theta"].grad = None
        E = autograd.energy(s["pos"], s["theta"], model, s["batch"], case["prec"])
        E.backward(s["gE"])
        out = [E.detach(), s["pos"].grad, s["theta"].grad]
        return out if case["prec"] == "fp64" else [v.float() for v in out]
    if kind == "active_set":
        api.mtp_set_active_set(model, s["A"])
        return api.mtp_get_active_inverse(model)
    if kind == "select":
        rows = api.mtp_param_rows(model, s["batch"], s["nbr"])
        A0 = torch.cat([rows[s["pick"]], s["gauge"] * rows.abs().max()])
        api.mtp_set_active_set(model, A0)
        source, swaps = api.mtp_maxvol(model, rows, eps=1e-2)
        return {"source": source, "swaps": swaps, "A": api.mtp_get_active_set(model), "rows": rows}
    near = api.mtp_extract_neighborhoods(s["nbr"], s["batch"], s["centers"])
    cluster = api.mtp_cut_clusters(s["batch"], s["centers"], case["radius"])
    return [_padded(near["off"], near["r"], near["type"]), _padded(cluster["off"], cluster["pos"], cluster["type"])]


def _padded(off, pos, species, room=320):
    """The batch form in which clusters are handed on: counts, positions and species [n, room]."""
    count = off[1:] - off[:-1]
    row = torch.repeat_interleave(torch.arange(len(count), device=off.device), count, output_size=len(species))
    slot = torch.arange(len(species), device=off.device) - off[row]
    x = pos.new_zeros((len(count), room, 3))
    z = torch.full((len(count), room), -1, dtype=species.dtype, device=off.device)
    x[row, slot], z[row, slot] = pos, species
    return [count, x, z]


def work(case):
    """Inputs read once and outputs written once; the multiply-adds of the method (the pairs of a
    neighborhood from the density, the contraction's terms from the model's sizes)."""
    kind = case["kind"]
    if kind == "cut":
        atoms = case["centers"] * 4.0 / 3.0 * math.pi * (5.0 ** 3 + case["radius"] ** 3) * 2 / 2.87 ** 3
        return {"bytes": atoms * (24 + 4 + 8), "flops": 10 * atoms}
    n_q = case.get("n_q", N_Q)
    z = api.mtp_describe(api.make_desc(case["types"], case["level"], n_q, R_MIN, case.get("r_cut", 5.0)))
    m = z["n_params"]
    if kind == "active_set":
        return {"bytes": 16.0 * m * m, "flops": 2.0 * m ** 3}
    rc3 = 4.0 / 3.0 * math.pi * case.get("r_cut", 5.0) ** 3
    if kind in ("train", "energy_grad"):
        n, pairs = case["n_cfg"] * (case["hi"] - 8) / math.log(case["hi"] / 8), rc3 * 0.086
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        lattice = case.get("lattice", "bcc")
        per, vol = {"fcc": (4, 3.6 ** 3), "bcc": (2, 2.87 ** 3), "liquid": (1024, 1024 / 0.085)}[lattice]
        n, pairs = cells * per - case.get("vacancies", 0), rc3 * per / vol
    # per pair: radial basis and functions, moments and their adjoint; per atom: the contraction
    mono = (z["nu_max"] + 1) * (z["nu_max"] + 2) * (z["nu_max"] + 3) // 6
    moments = 14 * N_Q + 4 * z["n_rad"] * N_Q + mono + 2 * z["n_mom_comps"]
    adjoint = 4 * z["n_mom_comps"] + 7 * mono + 2 * z["n_rad"] + 9
    rows = 2 * z["n_rad"] * N_Q
    flops = n * (pairs * (moments + adjoint) + 9 * z["n_triples"] + 2 * z["n_lin"])
    byts = n * (24 + 4)
    if kind == "md":
        byts += n * 32
        if case["grade"]:
            flops += n * (pairs * rows + 2.0 * m * m)
            byts += n * 8 + 8 * m * m
    elif kind == "train":           # the tangent of the rows: about two more passes
        flops = 3 * flops + n * pairs * 3 * rows
        byts += n * 24 + 8 * m
    elif kind == "energy_grad":
        flops += n * pairs * rows
        byts += n * 24 + 8 * m
    else:
        flops += n * pairs * rows + 2.0 * n * m * m + 2.0 * m ** 3
        byts = n * 28 + 8.0 * n * m + 16.0 * m * m
    return {"bytes": float(byts), "flops": float(flops)}


# ------------------------------------------------------------------------------------
# 64-bit values of the outputs, from the equations of the method in plain torch
# ------------------------------------------------------------------------------------

_PAIRS = {P: [(i, j) for i in range(P) for j in range(i + 1, P)] for P in range(1, 5)}


def _n_rad(level):
    return 1 + max(mu for labs, _ in _basis(level) for mu, _ in labs)


def _basis(level, _kept={}):
    """Basis functions up to `level` as (labels (mu, nu) per factor, edge multiplicities): contractions
    of at most four moments, none with itself, ordered by (level, factors, labels, smallest edges)."""
    if level in _kept:
        return _kept[level]
    lev = lambda lab: 2 + 4 * lab[0] + lab[1]   # noqa: E731
    labels = sorted((mu, nu) for mu in range(level) for nu in range(level) if lev((mu, nu)) <= level)
    found = set()

    def edges(left, pairs, got):
        if not pairs:
            if not any(left):
                yield tuple(got)
            return
        i, j = pairs[0]
        # the last pair of node i has to take what is left of it
        last = not any(i in p for p in pairs[1:])
        for e in ([left[i]] if last else range(min(left[i], left[j]) + 1)):
            if e <= min(left[i], left[j]):
                rest = list(left)
                rest[i] -= e
                rest[j] -= e
                yield from edges(rest, pairs[1:], got + [e])

    def multisets(P, start, room):
        if P == 0:
            yield ()
            return
        for k in range(start, len(labels)):
            if lev(labels[k]) + 2 * (P - 1) <= room:
                for rest in multisets(P - 1, k, room - lev(labels[k])):
                    yield (labels[k],) + rest

    for P in range(1, 5):
        perms = list(itertools.permutations(range(P)))
        at = {p: k for k, p in enumerate(_PAIRS[P])}
        for labs in multisets(P, 0, level):
            same = [p for p in perms if all(labs[p[k]] == labs[k] for k in range(P))]
            for e in edges([nu for _, nu in labs], _PAIRS[P], []):
                found.add((labs, min(tuple(e[at[tuple(sorted((p[i], p[j])))]] for i, j in _PAIRS[P]) for p in same)))
    _kept[level] = sorted(found, key=lambda f: (sum(map(lev, f[0])), len(f[0]), f[0], f[1]))
    return _kept[level]


def _pairs(b, r_cut, dev):
    """(i, j, r_ij) of every neighbor pair, by brute force over atoms and images."""
    out_i, out_j, out_r = [], [], []
    for k in range(len(b["atom_offset"]) - 1):
        a0, a1 = int(b["atom_offset"][k]), int(b["atom_offset"][k + 1])
        H = b["cell"][k]
        inv = np.linalg.inv(H)
        reach = np.ceil(r_cut * np.linalg.norm(inv, axis=0) + np.ptp(b["pos"][a0:a1] @ inv, axis=0)).astype(int)
        img = np.array(list(itertools.product(*(range(-n, n + 1) for n in reach))), float) @ H
        x = torch.as_tensor(b["pos"][a0:a1], device=dev)
        y = (x[:, None] + torch.as_tensor(img, device=dev)[None]).reshape(-1, 3)
        step = max(1, 60_000_000 // len(y))
        for c in range(0, a1 - a0, step):
            d2 = sum((y[None, :, q] - x[c:c + step, q, None]) ** 2 for q in range(3))
            i, p = torch.nonzero((d2 < r_cut * r_cut) & (d2 > 1e-16), as_tuple=True)
            i = i + c
            out_i.append(i + a0)
            out_j.append(torch.div(p, len(img), rounding_mode="floor") + a0)
            out_r.append(y[p] - x[i])
    return torch.cat(out_i), torch.cat(out_j), torch.cat(out_r)


class _Sites:
    """V_i and the basis values of neighborhoods as differentiable functions of r_ij and theta."""

    def __init__(self, case, dev):
        self.T, self.r_cut, self.dev = case["types"], case.get("r_cut", 5.0), dev
        self.basis = _basis(case["level"])
        self.NR, self.n_lin = _n_rad(case["level"]), len(self.basis)
        self.nu = {mu: max(nu for labs, _ in self.basis for m, nu in labs if m == mu) for mu in range(self.NR)}
        top = max(self.nu.values())
        self.mono = [(a, b, d - a - b) for d in range(top + 1) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]
        at = {e: k for k, e in enumerate(self.mono)}
        self.full = {}
        for d in range(top + 1):      # every index tuple of the rank-d tensor -> its monomial
            idx = [at[tuple(t.count(q) for q in range(3))] for t in itertools.product(range(3), repeat=d)]
            self.full[d] = torch.tensor(idx, device=dev)

    def radial(self, r):
        d = r.norm(dim=1)
        x = (2 * d - (R_MIN + self.r_cut)) / (self.r_cut - R_MIN)
        t = [torch.ones_like(x), x]
        while len(t) < N_Q:
            t.append(2 * x * t[-1] - t[-2])
        return torch.stack(t[:N_Q], 1) * ((self.r_cut - d) ** 2)[:, None]

    def values(self, f, r, i, n):
        """B[n, n_lin] from the radial functions f[pairs, NR] of the pairs of n centers."""
        pw = [torch.ones_like(r)]
        for _ in range(max(self.nu.values())):
            pw.append(pw[-1] * r)
        mono = torch.stack([pw[a][:, 0] * pw[b][:, 1] * pw[c][:, 2] for a, b, c in self.mono], 1)
        M = {}
        for mu, nu in self.nu.items():
            k = (nu + 1) * (nu + 2) * (nu + 3) // 6
            sums = torch.zeros((n, k), dtype=r.dtype, device=r.device).index_add(0, i, f[:, mu, None] * mono[:, :k])
            for d in range(nu + 1):
                M[mu, d] = sums[:, self.full[d]].reshape((n,) + (3,) * d)
        B = []
        for labs, e in self.basis:
            subs, free = [[] for _ in labs], iter("abcdefghijklmopqrstuvwxyz")
            for (p, q), count in zip(_PAIRS[len(labs)], e):
                for _ in range(count):
                    c = next(free)
                    subs[p].append(c)
                    subs[q].append(c)
            B.append(torch.einsum(",".join("n" + "".join(s) for s in subs) + "->n", *[M[lab] for lab in labs]))
        return torch.stack(B, 1)

    def f_of(self, c, Q, zi, zj):
        return torch.einsum("pmb,pb->pm", c[zi, zj], Q)

    def split(self, theta):
        T, n = self.T, self.n_lin
        return theta[:T], theta[T:T + n], theta[T + n:].reshape(T, T, self.NR, N_Q)


def _evaluate(case, b, theta, dev, want_rows, chunk):
    """V, dV_i/dr_ij, W_i and the rows b_i of every neighborhood, `chunk` centers at a time."""
    S = _Sites(case, dev)
    i, j, r = _pairs(b, S.r_cut, dev)
    z = torch.as_tensor(b["type"], device=dev).long()
    s, xi, c = S.split(torch.as_tensor(theta, device=dev))
    N = len(z)
    V, G, rows = torch.empty(N, dtype=r.dtype, device=dev), torch.empty_like(r), []
    ends = torch.searchsorted(i, torch.arange(0, N + chunk, chunk, device=dev).clamp(max=N)).tolist()
    for k, (p0, p1) in enumerate(zip(ends[:-1], ends[1:])):
        a0, a1 = k * chunk, min(N, (k + 1) * chunk)
        if a1 <= a0:
            break
        x = r[p0:p1].clone().requires_grad_(True)
        zi, zj, at = z[i[p0:p1]], z[j[p0:p1]], i[p0:p1] - a0
        Q = S.radial(x)
        f = S.f_of(c, Q, zi, zj)
        B = S.values(f, x, at, a1 - a0)
        v = B @ xi
        V[a0:a1] = (v + s[z[a0:a1]]).detach()
        g, gf = torch.autograd.grad(v.sum(), (x, f))
        G[p0:p1] = g
        if want_rows:
            n = a1 - a0
            own = torch.zeros((n * S.T, S.NR * N_Q), dtype=r.dtype, device=dev)
            own.index_add_(0, at * S.T + zj, (gf[:, :, None] * Q.detach()[:, None, :]).reshape(len(gf), -1))
            cb = torch.zeros((n, S.T, S.T * S.NR * N_Q), dtype=r.dtype, device=dev)
            cb[torch.arange(n, device=dev), z[a0:a1]] = own.reshape(n, -1)
            one = torch.nn.functional.one_hot(z[a0:a1], S.T).to(r.dtype)
            rows.append(torch.cat([one, B.detach(), cb.reshape(n, -1)], 1))
    F = torch.zeros((N, 3), dtype=r.dtype, device=dev).index_add(0, i, G).index_add(0, j, -G)
    W = -G[:, :, None] * r[:, None, :]
    cfg = torch.as_tensor(np.repeat(np.arange(len(b["atom_offset"]) - 1), np.diff(b["atom_offset"])), device=dev)
    K = len(b["atom_offset"]) - 1
    E = torch.zeros(K, dtype=r.dtype, device=dev).index_add(0, cfg, V)
    W = torch.zeros((K, 3, 3), dtype=r.dtype, device=dev).index_add(0, cfg[i], W)
    return E, V, F, W, cfg, (torch.cat(rows) if want_rows else None)


def _loss_grad(case, x, dev):
    b, S = x["batch"], _Sites(case, dev)
    theta = torch.as_tensor(x["theta"], device=dev).requires_grad_(True)
    ref = {k: torch.as_tensor(x[k], device=dev) for k in ("E_ref", "F_ref", "W_ref")}
    w_s, total, grad = (1e-3 if case["stress"] else 0.0), 0.0, torch.zeros_like(theta)
    ao = b["atom_offset"]
    for k0 in range(0, case["n_cfg"], 32):
        k1 = min(case["n_cfg"], k0 + 32)
        a0, a1 = int(ao[k0]), int(ao[k1])
        part = {"atom_offset": ao[k0:k1 + 1] - a0, "pos": b["pos"][a0:a1], "cell": b["cell"][k0:k1]}
        i, j, r = _pairs(part, S.r_cut, dev)
        z = torch.as_tensor(b["type"][a0:a1], device=dev).long()
        cfg = torch.as_tensor(np.repeat(np.arange(k1 - k0), np.diff(part["atom_offset"])), device=dev)
        s, xi, c = S.split(theta)
        r.requires_grad_(True)
        f = S.f_of(c, S.radial(r), z[i], z[j])
        V = S.values(f, r, i, a1 - a0) @ xi + s[z]
        (G,) = torch.autograd.grad(V.sum(), r, create_graph=True)
        E = torch.zeros(k1 - k0, dtype=V.dtype, device=dev).index_add(0, cfg, V)
        F = torch.zeros((a1 - a0, 3), dtype=V.dtype, device=dev).index_add(0, i, G).index_add(0, j, -G)
        W = torch.zeros((k1 - k0, 9), dtype=V.dtype, device=dev)
        W = W.index_add(0, cfg[i], -(G[:, :, None] * r.detach()[:, None, :]).reshape(-1, 9))
        L = ((E - ref["E_ref"][k0:k1]) ** 2).sum() + 0.01 * ((F - ref["F_ref"][a0:a1]) ** 2).sum()
        L = L + w_s * ((W - ref["W_ref"][k0:k1]) ** 2).sum()
        grad += torch.autograd.grad(L, theta)[0]
        total += float(L.detach())
    return [torch.tensor([total], dtype=torch.float64), grad]


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "md":
        cells = case["nx"] * case["ny"] * case["nz"]
        if case["lattice"] == "liquid" or cells * len(LATTICES[case["lattice"]][0]) > 20000:
            return None
    x = _inputs(case, seed)
    if kind == "active_set":
        return torch.linalg.inv(torch.as_tensor(x["A"], device=dev))
    if kind == "train":
        return _loss_grad(case, x, dev)
    if kind == "md":
        E, V, F, W, _, rows = _evaluate(case, x["batch"], x["theta"], dev, case["grade"], 1024)
        out = {"energy": E, "site_energy": V, "forces": F, "virial": W}
        if case["grade"]:
            out["gamma"] = torch.linalg.solve(torch.as_tensor(x["A"], device=dev), rows, left=False).abs().amax(1)
        return out
    if kind == "energy_grad":
        E, _, F, _, cfg, rows = _evaluate(case, x["batch"], x["theta"], dev, True, 1024)
        gE = torch.as_tensor(x["gE"], device=dev)
        return [E, -gE[cfg, None] * F, gE[cfg] @ rows]
    if kind == "select":
        rows = _evaluate(case, x["batch"], x["theta"], dev, True, 1024)[5]
        return {"source": None, "swaps": None, "A": None, "rows": rows}
    return None     # cut: indices and copied positions
