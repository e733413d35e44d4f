"""dL/dc at the edges of its kernel: four atoms of eight lanes at a time, chunks of atoms sorted by species.

Species counts up to 8, radial sizes that are and are not known at compile time, single atoms, atom
counts that leave slots empty, and batches large enough for chunks of more than four atoms (compared with
the sum over smaller batches: the loss is a sum over configurations).  Tolerances: the existing ones of
the double path (1e-8 against the oracle); 1e-10 of the largest entry between two device sums.
"""

import numpy as np
import pytest
import torch

import oracle
from oracle import levels, loss as oloss
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu

W = (1.0, 0.01, 0.001)


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _params(L, S, NQ, seed):
    labels = synth.labels_from_level_table(levels.level_table(L))
    return synth.scaled_params(L, S, NQ, 1.0, 5.0, labels, seed=seed, radial_decay=0.5)


def _batch(sizes, S, seed):
    rng = np.random.default_rng(seed)
    cfgs = []
    for n in sizes:
        c = synth.random_small_config(rng, n, n, species_pool=tuple(range(S)), max_species=S)
        c.types[:] = rng.integers(0, S, size=c.n)
        cfgs.append(c)
    return cfgs, synth.pack(cfgs), rng


def _grad(model, b, refs):
    return [t.cpu().numpy() for t in model.param_grad(dev(b.pos), dev(b.types, torch.int32), dev(b.cells),
                                                       dev(b.cfg_off, torch.int32), *map(dev, refs), W)]


@pytest.mark.parametrize("L,S,NQ,sizes", [(6, 1, 8, [1]), (8, 3, 8, [1, 2, 5, 9]), (8, 2, 7, [3, 6]),
                                          (10, 8, 16, [7, 12]), (20, 2, 5, [6])])
def test_against_the_oracle(gpu_lib, L, S, NQ, sizes):
    p = _params(L, S, NQ, 3)
    cfgs, b, rng = _batch(sizes, S, 11 * L + S)
    refs = (rng.normal(size=b.n_cfg), rng.normal(size=(b.n_atoms, 3)), rng.normal(size=(b.n_cfg, 9)))
    loss, dxi, dc = _grad(mtp.Model.from_params(p, "fp64"), b, refs)
    ref = [dict(energy=refs[0][k], forces=refs[1][b.cfg_off[k]:b.cfg_off[k + 1]], virial=refs[2][k].reshape(3, 3))
           for k in range(b.n_cfg)]
    pot = oracle.Potential(p)
    for q in range(2):
        vxi, vc = rng.normal(size=dxi.shape) * (q == 0) * np.abs(p.xi), rng.normal(size=dc.shape)
        L0, dL = oloss.loss_and_directional(pot, cfgs, ref, W, "vibrations", p.xi, p.c, vxi, vc)
        scale = np.abs(dxi * vxi).sum() + np.abs(dc * vc).sum()
        assert abs(np.dot(dxi, vxi) + np.sum(dc * vc) - dL) <= 1e-8 * max(abs(dL), scale)
        assert loss[0] == pytest.approx(L0, rel=1e-10)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("S,NQ", [(3, 8), (2, 6)])
def test_large_batches_are_sums_of_small_ones(gpu_lib, precision, tol, S, NQ):
    p = _params(10, S, NQ, 5)
    sizes = [int(n) for n in np.random.default_rng(1).integers(8, 64, size=331)]
    cfgs, b, rng = _batch(sizes, S, 17)
    assert b.n_atoms > 8000  # chunks of eight atoms
    refs = (rng.normal(size=b.n_cfg), rng.normal(size=(b.n_atoms, 3)), rng.normal(size=(b.n_cfg, 9)))
    model = mtp.Model.from_params(p, precision)
    whole = _grad(model, b, refs)
    parts = [0.0, 0.0, 0.0]
    for lo in range(0, b.n_cfg, 67):
        hi = min(b.n_cfg, lo + 67)
        q = synth.pack(cfgs[lo:hi])
        i0, i1 = int(b.cfg_off[lo]), int(b.cfg_off[hi])
        parts = [x + y for x, y in zip(parts, _grad(model, q, (refs[0][lo:hi], refs[1][i0:i1], refs[2][lo:hi])))]
    for x, y in zip(whole, parts):
        assert np.abs(x - y).max() <= tol * np.abs(y).max()
