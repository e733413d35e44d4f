"""What is timed: the calls a user of the MTP library makes, over the sizes they make them at.

Kinds of case (each through the public binding, `paper_2007_08555_gb300.mtp.Model`):
  eval    energy, forces and virial of a batch, neighbour search included (Model.eval_batch)
  grad    training loss and its gradient in theta = {xi, c} (Model.param_grad)
  md      velocity-Verlet steps with a skin list (Model.md_run)
  relax   FIRE over positions and cells (Model.relax_batch)
  grade   extrapolation grades of given rows (Model.grade)
  select  MaxVol selection of an active set, and the grades of all its candidates
          (Model.select_active_set, Model.grade)

Inputs follow the recipes of `synth.py` (fcc 3.6, bcc 3.2, hcp 2.55 Angstrom; Gaussian displacements;
random species; R_cut = 5, N_Q = 8).  xi is scaled per basis function (`synth.scaled_params`), so that
every basis function contributes, as in a fitted potential.  Single crystals take R_min = 2 and a few pairs
fall below it; the noisy random cells, training, relaxation and MD take the smooth radial recipe (R_min = 1,
coefficients damped by 0.5^b).

The float path writes float results into double arrays.  A program that chose it keeps them as float, and
so does run(): the outputs' type is then that of the arithmetic.  The double path's stay double.
"""

import functools
import math

import numpy as np
import torch

from paper_2007_08555_gb300 import flops, mtp, synth

R_CUT, N_Q = 5.0, 8
MASSES = np.array([26.98, 58.69, 63.55])  # amu
BASIS = {8: 9, 10: 17, 12: 32, 14: 61, 16: 116, 18: 229, 20: 460}  # basis functions of a level
LATTICE_CELLS = {"fcc": 4, "bcc": 2, "hcp": 2}  # atoms of the conventional cell


# -- the cases ------------------------------------------------------------------------------------
def listed():
    return [
        # one small cell at a low level: the call of an interactive program or of a small-cell MD code,
        # where launches and waits are what it costs
        dict(name="eval_bcc128_lev10", kind="eval", cells="bcc", reps=4, sigma=0.1, lev=10, species=1,
             precision="fp32"),
        # an ordinary simulation cell at the level of fitted alloy potentials
        dict(name="eval_fcc16k_lev16", kind="eval", cells="fcc", reps=16, sigma=0.15, lev=16, species=2,
             precision="fp32"),
        # the largest: one evaluation of a million-atom alloy at the highest level
        dict(name="eval_fcc1m_lev20", kind="eval", cells="fcc", reps=64, sigma=0.1, lev=20, species=3,
             precision="fp32"),
        # screening of thousands of small ragged cells in one call
        dict(name="eval_cells4096_lev16", kind="eval", cells="random", n_cfg=4096, n_lo=8, n_hi=256, lev=16,
             species=3, precision="fp32"),
        # the same in double precision, fewer of them: reference energies of candidate structures
        dict(name="eval_cells509_lev16_f64", kind="eval", cells="random", n_cfg=509, n_lo=8, n_hi=256, lev=16,
             species=3, precision="fp64"),
        # one step of training on a large set of labelled cells
        dict(name="grad_cells2048_lev20", kind="grad", n_cfg=2048, n_lo=32, n_hi=128, lev=20, species=3,
             precision="fp32", scaling="vibrations"),
        # one step of training on a small set in double precision, as in the first rounds of active learning
        dict(name="grad_cells67_lev12_f64", kind="grad", n_cfg=67, n_lo=16, n_hi=128, lev=12, species=2,
             precision="fp64", scaling="structures"),
        # a stretch of molecular dynamics of an ordinary cell
        dict(name="md_fcc16k_lev16", kind="md", reps=16, lev=16, species=3, steps=10, precision="fp32"),
        # relaxation of candidate structures, positions and cells
        dict(name="relax_cells61_lev12", kind="relax", n_cfg=61, n_lo=8, n_hi=96, lev=12, species=2, steps=20,
             precision="fp32"),
        # per-atom grades of a large cell or batch: the rows are there, the tensor-core grade runs alone
        dict(name="grade_300k_m116", kind="grade", rows=300_007, lev=16, precision="fp32_tc"),
        # the active set of the first 2 m candidates at an ordinary and at the highest level
        dict(name="select_232_m116", kind="select", rows=232, lev=16, precision="fp64"),
        dict(name="select_920_m460", kind="select", rows=920, lev=20, precision="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "batch", "batch", "f64", "grad", "grad", "gradf64", "md", "relax", "grade",
                       "select"])
    lev = rng.choice([8, 10, 12, 14, 16, 18, 20])
    if kind == "eval":
        cells = rng.choice(["fcc", "bcc", "hcp"])
        reps = _log(rng, 2, 48)
        return dict(kind="eval", cells=cells, reps=reps, sigma=round(rng.uniform(0.05, 0.2), 3), lev=lev,
                    species=rng.randint(1, 3), precision="fp32")
    if kind in ("batch", "f64"):
        f64 = kind == "f64"
        lo = _log(rng, 2, 24)
        return dict(kind="eval", cells="random", n_cfg=_log(rng, 3, 350 if f64 else 4096), n_lo=lo,
                    n_hi=lo + _log(rng, 8, 200), lev=min(lev, 16) if f64 else lev, species=rng.randint(1, 3),
                    precision="fp64" if f64 else "fp32")
    if kind in ("grad", "gradf64"):
        f64 = kind == "gradf64"
        lo = _log(rng, 8, 32)
        return dict(kind="grad", n_cfg=_log(rng, 5, 67 if f64 else 2048), n_lo=lo, n_hi=lo + _log(rng, 8, 96),
                    lev=min(lev, 12) if f64 else lev, species=rng.randint(1, 3 if not f64 else 2),
                    precision="fp64" if f64 else "fp32",
                    scaling=rng.choice(["vibrations", "structures", "molecules"]))
    if kind == "md":
        return dict(kind="md", reps=rng.randint(4, 16), lev=min(lev, 16), species=rng.randint(1, 3),
                    steps=rng.randint(3, 10), precision="fp32")
    if kind == "relax":
        lo = _log(rng, 4, 16)
        return dict(kind="relax", n_cfg=_log(rng, 3, 61), n_lo=lo, n_hi=lo + _log(rng, 8, 80), lev=min(lev, 12),
                    species=rng.randint(1, 2), steps=rng.randint(8, 20), precision="fp32")
    if kind == "grade":
        lev = max(lev, 12)
        return dict(kind="grade", rows=_log(rng, 50, min(300_000, 300_000 * 116 ** 2 // BASIS[lev] ** 2)), lev=lev,
                    precision="fp32_tc")
    lev = max(lev, 10)
    m = BASIS[lev]
    return dict(kind="select", rows=m + rng.randint(1, m), lev=lev, precision="fp64")


# -- inputs ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _repetitions(n_target, per_cell):
    """Near-cubic repetition of a cell of per_cell atoms with at least n_target atoms."""
    best = None
    side = int((n_target / per_cell) ** (1 / 3)) + 2
    for a in range(1, side + 2):
        for b in range(1, a + 1):
            for c in range(1, b + 1):
                n = per_cell * a * b * c
                if n >= n_target and (best is None or (n, a / c) < best[0]):
                    best = ((n, a / c), (c, b, a))
    return best[1]


@functools.lru_cache(maxsize=None)
def _block(kind, reps):
    return synth.supercell(synth.LATTICES[kind](), reps)


def _random_cells(rng, n_cfg, n_lo, n_hi, species):
    """Strained, displaced fcc/bcc/hcp cells with vacancies, atom counts log-uniform (synth.py's recipe)."""
    pos, types, cells, off = [], [], [], [0]
    # the atom counts belong to the case: the same for every seed
    sizes = np.random.default_rng([n_cfg, n_lo, n_hi]).uniform(math.log(n_lo), math.log(n_hi), size=n_cfg)
    for n in np.rint(np.exp(sizes)).astype(int).tolist():
        kind = ("fcc", "bcc", "hcp")[rng.integers(3)]
        x, H = _block(kind, _repetitions(n, LATTICE_CELLS[kind]))
        x = x[np.sort(rng.permutation(x.shape[0])[:n])]
        e = rng.uniform(-0.05, 0.05, size=(3, 3))
        strain = np.eye(3) + 0.5 * (e + e.T)
        pos.append(x @ strain.T + rng.normal(0.0, rng.uniform(0.1, 0.3), size=x.shape))
        cells.append(H @ strain.T)
        some = rng.permutation(species)[:rng.integers(1, species + 1)]
        types.append(some[rng.integers(0, some.size, size=n)])
        off.append(off[-1] + n)
    return (np.concatenate(pos), np.concatenate(types).astype(np.int32), np.stack(cells),
            np.array(off, dtype=np.int32))


def _structures(case, rng):
    if case.get("cells") in LATTICE_CELLS:  # one large cell
        r = case["reps"]
        x, H = _block(case["cells"], (r, r, r))
        x = x + rng.normal(0.0, case["sigma"], size=x.shape)
        return (x, rng.integers(0, case["species"], size=x.shape[0]).astype(np.int32), H[None],
                np.array([0, x.shape[0]], dtype=np.int32))
    return _random_cells(rng, case["n_cfg"], case["n_lo"], case["n_hi"], case["species"])


def _r_min(case):
    return 2.0 if case.get("cells") in LATTICE_CELLS else 1.0


def _potential(case, seed, table):
    smooth = case.get("cells") not in LATTICE_CELLS
    p = synth.scaled_params(case["lev"], case["species"], N_Q, _r_min(case), R_CUT,
                            synth.labels_from_level_table(table), seed, radial_decay=0.5 if smooth else 1.0)
    # the cohesive energy of a fitted potential, about -3 eV per atom, in the first basis function, M_{0,0};
    # for relaxation a soft repulsion, since random parameters hold no cell up
    p.c[:, :, 0, 0] = 0.3
    p.xi[0] = 0.02 if case["kind"] == "relax" else -0.1
    return p


def _arrays(case, seed):
    """Every input of an evaluating case as numpy arrays, from the seed alone."""
    rng = np.random.default_rng([seed, 1])
    if case["kind"] == "md":
        x, types, H, off = _structures(dict(case, cells="fcc", sigma=0.02), rng)
        vel = synth.maxwell_velocities(types, MASSES, 300.0, seed)
        return dict(pos=x, types=types, cells=H, off=off, vel=vel)
    pos, types, cells, off = _structures(case, rng)
    a = dict(pos=pos, types=types, cells=cells, off=off)
    if case["kind"] == "grad":
        n = np.diff(off).astype(np.float64)
        a["e_ref"] = n * rng.normal(0.0, 0.1, size=n.size)
        a["f_ref"] = rng.normal(0.0, 0.5, size=pos.shape)
        a["w_ref"] = np.sqrt(n)[:, None] * rng.normal(0.0, 0.5, size=(n.size, 9))
    return a


def _rows(n, m, rng):
    """Rows like b(cfg): columns over nine decades."""
    return torch.randn((n, m), dtype=torch.float64, device="cuda", generator=rng) * torch.logspace(
        -3, 6, m, dtype=torch.float64, device="cuda")


def _row_inputs(case, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    m = BASIS[case["lev"]]
    return _rows(m, m, g) if case["kind"] == "grade" else None, _rows(case["rows"], m, g)


def prepare(case, seed):
    if case["kind"] in ("grade", "select"):
        A, rows = _row_inputs(case, seed)
        model = mtp.Model(case["lev"], 1, N_Q, 2.0, R_CUT, precision=case["precision"])
        if A is not None:
            mtp.mtp_set_active_set(model.h, A.cpu().numpy())
        return dict(case=case, model=model, rows=rows)
    a = _arrays(case, seed)
    model = mtp.Model(case["lev"], case["species"], N_Q, _r_min(case), R_CUT, precision=case["precision"])
    p = _potential(case, seed, model.level_table())
    model.set_params(p.xi, p.c)
    if case["kind"] == "md":
        model.set_skin(0.5)
    s = {k: torch.as_tensor(np.ascontiguousarray(v), device="cuda") for k, v in a.items()}
    return dict(case=case, model=model, **s)


# -- one pass -------------------------------------------------------------------------------------
def run(s):
    case, model = s["case"], s["model"]
    kept = torch.float64 if case["precision"] == "fp64" else torch.float32
    kind = case["kind"]
    if kind == "eval":
        out = model.eval_batch(s["pos"], s["types"], s["cells"], s["off"])
        return {k: out[k].to(kept) for k in ("energy", "forces", "virial")}
    if kind == "grad":
        loss, dxi, dc = model.param_grad(s["pos"], s["types"], s["cells"], s["off"], s["e_ref"], s["f_ref"],
                                         s["w_ref"], scaling=case["scaling"])
        return {"loss": loss.to(kept), "dxi": dxi.to(kept), "dc": dc.to(kept)}
    if kind == "md":
        x, v = s["pos"].clone(), s["vel"].clone()
        e_pot, e_kin, rebuilds = model.md_run(x, v, s["types"], s["cells"], MASSES[:case["species"]], 1.0,
                                              case["steps"])
        return {"pos": x.to(kept), "vel": v.to(kept), "e_pot": e_pot.astype(np.float32),
                "e_kin": e_kin.astype(np.float32), "rebuilds": rebuilds}
    if kind == "relax":
        x, H = s["pos"].clone(), s["cells"].clone()
        # small steps: the first ones of noisy structures, far from their minimum
        energy, steps, status = model.relax_batch(x, s["types"], H, s["off"], max_steps=case["steps"], dt=0.005,
                                                  dt_max=0.02)
        return {"pos": x.to(kept), "cells": H.to(kept), "energy": energy.to(kept), "steps": steps, "status": status}
    if kind == "grade":
        return {"gamma": model.grade(s["rows"])}
    rows, swaps, largest = model.select_active_set(s["rows"])
    return {"rows": rows, "swaps": swaps, "largest": largest, "gamma": model.grade(s["rows"])}


# -- what a pass cannot do without ----------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _per_unit(lev):
    return flops.counts(lev, N_Q)


def work(case):
    if case["kind"] in ("grade", "select"):
        n, m = case["rows"], BASIS[case["lev"]]
        if case["kind"] == "grade":  # the rows and A^-1 read, the grades written; b A^-1
            return {"bytes": 8 * (n * m + m * m + n), "flops": 2 * n * m * m}
        # elimination of the tall matrix, an inverse, C = B A^-1 for the selection
        return {"bytes": 8 * (n * m + m * m + n), "flops": 2 * n * m * m - 2 * m ** 3 // 3 + 2 * m ** 3 + 2 * n * m * m}
    if case["kind"] == "md" or case.get("cells") in LATTICE_CELLS:
        cell = case.get("cells", "fcc")
        n, k = LATTICE_CELLS[cell] * case["reps"] ** 3, 1
    else:
        k, lo, hi = case["n_cfg"], case["n_lo"], case["n_hi"]
        n = int(k * (hi - lo) / math.log(hi / lo))  # mean of the log-uniform atom counts
    pairs = 42 * n
    u = _per_unit(case["lev"])
    once = (u["pair_moments"] + u["pair_adjoint"] + u["pair_gather"]) * pairs + u["atom_contract"] * n
    # positions (and velocities), species and cells in; energies, forces and virials out
    io = n * (24 + 4 + 24) + k * (72 + 8 + 72)
    if case["kind"] == "grad":
        # the evaluation, and its derivative along the residuals: moments' tangent, contraction on
        # (value, tangent) pairs, and the pairs' shares of dL/dc
        return {"bytes": io + n * 24 + k * 80,
                "flops": once + (2 * u["pair_moments"] + u["pair_adjoint"]) * pairs + 3 * u["atom_contract"] * n}
    if case["kind"] == "md":
        return {"bytes": n * (24 + 24 + 4 + 24 + 24), "flops": once * (case["steps"] + 1)}
    if case["kind"] == "relax":
        return {"bytes": n * (24 + 4 + 24) + k * (144 + 16), "flops": once * (case["steps"] + 1)}
    return {"bytes": io, "flops": once}


# -- the same in 64 bits, from the definitions ----------------------------------------------------
def _graphs(table):
    """The basis functions of a level table: lists of components (nodes (mu, nu), adjacency)."""
    t, at, out = [int(v) for v in table], 1, []
    for _ in range(t[0]):
        n_comp, at, comps = t[at + 1], at + 2, []
        for _ in range(n_comp):
            n = t[at]
            nodes = tuple((t[at + 1 + 2 * q], t[at + 2 + 2 * q]) for q in range(n))
            at += 1 + 2 * n
            edges = tuple(t[at:at + n * (n - 1) // 2])
            at += n * (n - 1) // 2
            comps.append((nodes, edges))
        out.append(comps)
    return out


def _contract(nodes, edges, M):
    """One connected contraction of moment tensors M[(mu, nu)] [atoms, 3, ..., 3]."""
    n = len(nodes)
    letters = [[] for _ in nodes]
    q, free = 0, "abcdefghijklmnopqrstuvwxy"
    for u in range(n):
        for v in range(u + 1, n):
            for _ in range(edges[q]):
                letters[u].append(free[0])
                letters[v].append(free[0])
                free = free[1:]
            q += 1
    left = list(range(1, n))
    have, T = letters[0], M[nodes[0]]
    while left:  # next the neighbour that leaves the fewest open indices
        v = min((w for w in left if set(letters[w]) & set(have) or not have), key=lambda w: len(
            set(letters[w]) ^ set(have)))
        left.remove(v)
        new = [c for c in have if c not in letters[v]] + [c for c in letters[v] if c not in have]
        T = torch.einsum("z%s,z%s->z%s" % ("".join(have), "".join(letters[v]), "".join(new)), T, M[nodes[v]])
        have = new
    return T


def _site_energies(r, zi, zj, present, xi, c, graphs, r_min):
    """V_i of padded neighbourhoods: r [atoms, most, 3], species zi [atoms], zj [atoms, most]."""
    d = torch.sqrt((r * r).sum(-1))
    x = (2 * d - r_min - R_CUT) / (R_CUT - r_min)
    T = [torch.ones_like(x), x]
    while len(T) < N_Q:
        T.append(2 * x * T[-1] - T[-2])
    Q = torch.stack(T[:N_Q], -1) * ((R_CUT - d) ** 2 * present)[..., None]
    f = (c[zi[:, None], zj] * Q[:, :, None, :]).sum(-1)  # [atoms, most, N_mu]
    labels = sorted({lab for comps in graphs for nodes, _ in comps for lab in nodes})
    M, mono = {}, torch.ones_like(d)[..., None]  # mono: r x ... x r, flattened
    for nu in range(max(nu for _, nu in labels) + 1):
        mus = [mu for mu, k in labels if k == nu]
        if mus:
            t = torch.bmm(f[:, :, mus].transpose(1, 2), mono)
            for k, mu in enumerate(mus):
                M[(mu, nu)] = t[:, k].reshape((-1,) + (3,) * nu)
        mono = (mono[..., None] * r[:, :, None, :]).reshape(*d.shape, -1)
    value, V = {}, 0.0
    for alpha, comps in enumerate(graphs):
        B = xi[alpha]
        for comp in comps:
            if comp not in value:
                value[comp] = _contract(*comp, M)
            B = B * value[comp]
        V = V + B
    return V


def _pairs(pos, H):
    """Pairs (i, j, s H) of one periodic cell within R_CUT."""
    n = pos.shape[0]
    inverse = np.linalg.inv(H)
    width = 1.0 / np.linalg.norm(inverse, axis=0)  # between opposite faces
    H, inv = torch.as_tensor(H, device=pos.device), torch.as_tensor(inverse, device=pos.device)
    frac = pos @ inv
    wrap = torch.floor(frac)
    x = (frac - wrap) @ H
    reach = [int(math.ceil(R_CUT / w)) for w in width]
    shifts = torch.cartesian_prod(*[torch.arange(-k, k + 1, device=pos.device) for k in reach]).double()
    rows = max(1, int(2e7 // (n * len(shifts))))
    if width.min() > 2.2 * R_CUT:  # the nearest image is the only one
        rows, shifts = max(1, int(2e7 // n)), None
    I, J, S = [], [], []
    for a in range(0, n, rows):
        d = x[None] - x[a:a + rows, None]
        if shifts is None:
            s = -torch.round(d @ inv)
            q = torch.nonzero(((d + s @ H) ** 2).sum(-1) < R_CUT ** 2)
            q = q[q[:, 0] + a != q[:, 1]]
            s = s[q[:, 0], q[:, 1]]
        else:
            e = d[:, :, None] + (shifts @ H)[None, None]
            q = torch.nonzero((e * e).sum(-1) < R_CUT ** 2)
            q = q[(q[:, 0] + a != q[:, 1]) | (shifts[q[:, 2]] != 0).any(-1)]
            s = shifts[q[:, 2]]
        i, j = q[:, 0] + a, q[:, 1]
        I.append(i)
        J.append(j)
        S.append(s + wrap[i] - wrap[j])
    return torch.cat(I), torch.cat(J), torch.cat(S) @ H


def _neighbourhoods(a):
    """Padded neighbour lists of a batch: j, s H and presence [atoms, most]."""
    I, J, S = [], [], []
    off, cells = a["off"].tolist(), a["cells"].cpu().numpy()
    for k, (lo, hi) in enumerate(zip(off, off[1:])):
        i, j, s = _pairs(a["pos"][lo:hi], cells[k])
        I.append(i + lo)
        J.append(j + lo)
        S.append(s)
    I, J, S = torch.cat(I), torch.cat(J), torch.cat(S)
    order = torch.argsort(I, stable=True)
    I, J, S = I[order], J[order], S[order]
    n = a["pos"].shape[0]
    count = torch.bincount(I, minlength=n)
    most = max(1, int(count.max()))
    slot = torch.arange(I.numel(), device=I.device) - (torch.cumsum(count, 0) - count)[I]
    j = torch.arange(n, device=I.device)[:, None].repeat(1, most)  # an absent neighbour is the atom itself
    sh = torch.full((n, most, 3), 4.0, dtype=torch.float64, device=I.device)
    there = torch.zeros((n, most), dtype=torch.float64, device=I.device)
    j[I, slot], sh[I, slot], there[I, slot] = J, S, 1.0
    return j, sh, there


def _cost(case):
    """Atoms times their largest tensor times the contractions: what exact() takes time for."""
    return work(case)["bytes"] / 52 * 3 ** (case["lev"] // 2 - 2) * BASIS[case["lev"]]


def exact(case, seed):
    if case["kind"] == "grade":
        A, rows = _row_inputs(case, seed)
        scale = 1.0 / A.abs().amax(0)  # equilibrated columns change nothing in b A^-1 but its rounding
        C = (rows * scale) @ torch.linalg.inv(A * scale)
        return {"gamma": C.abs().amax(1)}
    if case["kind"] == "select":
        rows = _row_inputs(case, seed)[1].cpu().numpy()
        C, largest = _maxvol(rows)
        return {"rows": None, "swaps": None, "largest": largest, "gamma": np.abs(C).max(1)}
    if case["kind"] in ("md", "relax") or _cost(case) > (3e10 if case["kind"] == "eval" else 3e9):
        return None
    a = {k: torch.as_tensor(np.ascontiguousarray(v), device="cuda") for k, v in _arrays(case, seed).items()}
    table = mtp.Model(case["lev"], case["species"], N_Q, 1.0, R_CUT).level_table()  # the order of xi
    p = _potential(case, seed, table)
    xi, c = torch.as_tensor(p.xi, device="cuda"), torch.as_tensor(p.c, device="cuda")
    j, sh, there = _neighbourhoods(a)
    graphs, z = _graphs(table), a["types"].long()
    k_of = torch.repeat_interleave(torch.arange(a["cells"].shape[0], device="cuda"), torch.diff(a["off"].long()))
    chunk = max(16, int(4e7 // (j.shape[1] * 3 ** (case["lev"] // 2 - 2))))
    if case["kind"] == "eval":
        n, K = a["pos"].shape[0], a["cells"].shape[0]
        E, F, W = (torch.zeros(s, dtype=torch.float64, device="cuda") for s in ((K,), (n, 3), (K, 3, 3)))
        for lo in range(0, n, chunk):
            q = slice(lo, min(n, lo + chunk))
            r = (a["pos"][j[q]] + sh[q] - a["pos"][q][:, None]).requires_grad_()
            V = _site_energies(r, z[q], z[j[q]], there[q], xi, c, graphs, p.r_min)
            (g,) = torch.autograd.grad(V.sum(), r)
            E.index_add_(0, k_of[q], V.detach())
            F[q] += g.sum(1)
            F.index_add_(0, j[q].reshape(-1), -g.reshape(-1, 3))
            W.index_add_(0, k_of[q], -torch.einsum("anu,anv->auv", g, r.detach()))
        return {"energy": E, "forces": F, "virial": W}
    # the loss (energy weight 1, forces 0.01, virial 0.001) and its gradient, a few configurations at a time
    xi.requires_grad_()
    c.requires_grad_()
    loss, dxi, dc = 0.0, 0.0, 0.0
    off, k = a["off"].tolist(), 0
    while k < len(off) - 1:
        k1 = k + 1
        while k1 < len(off) - 1 and off[k1 + 1] - off[k] <= chunk:
            k1 += 1
        q = slice(off[k], off[k1])
        r = (a["pos"][j[q]] + sh[q] - a["pos"][q][:, None]).requires_grad_()
        V = _site_energies(r, z[q], z[j[q]], there[q], xi, c, graphs, p.r_min)
        (g,) = torch.autograd.grad(V.sum(), r, create_graph=True)
        kk, size = k_of[q] - k, torch.diff(a["off"][k:k1 + 1].double())
        new = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
        E = new(k1 - k).index_add(0, kk, V)
        F = g.sum(1).index_add(0, j[q].reshape(-1) - off[k], -g.reshape(-1, 3))
        W = new(k1 - k, 3, 3).index_add(0, kk, -torch.einsum("anu,anv->auv", g, r))
        se, sf, ss = {"molecules": (size ** 0, size ** 0, size ** 0), "structures": (size ** -2, 1 / size, size ** -2),
                      "vibrations": (1 / size, size ** 0, 1 / size)}[case["scaling"]]
        L = ((se * (E - a["e_ref"][k:k1]) ** 2).sum() +
             0.01 * (sf[kk] * ((F - a["f_ref"][q]) ** 2).sum(-1)).sum() +
             0.001 * (ss * ((W.reshape(-1, 9) - a["w_ref"][k:k1]) ** 2).sum(-1)).sum())
        g_xi, g_c = torch.autograd.grad(L, (xi, c))
        loss, dxi, dc = loss + L.detach(), dxi + g_xi, dc + g_c
        k = k1
    return {"loss": loss.reshape(1), "dxi": dxi, "dc": dc}


def _maxvol(B):
    """C = B A^-1 of the MaxVol selection (start: pivot rows of an LU; swaps while |C| > 1.001)."""
    B = B / np.abs(B).max(0)
    n, m = B.shape
    W, order = B.copy(), np.arange(n)
    for k in range(m):
        p = k + int(np.argmax(np.abs(W[order[k:], k])))
        order[[k, p]] = order[[p, k]]
        rest, top = order[k + 1:], order[k]
        W[rest, k:] -= np.outer(W[rest, k] / W[top, k], W[top, k:])
    C = B @ np.linalg.inv(B[order[:m]])
    for _ in range(100 * m):
        k, j = divmod(int(np.argmax(np.abs(C))), m)
        if abs(C[k, j]) <= 1.001:
            break
        row = C[k].copy()
        row[j] -= 1.0
        C -= np.outer(C[:, j] / C[k, j], row)
    return C, float(np.abs(C).max())
