"""Reverse-pair slots: forces against the oracle where the search's tiles of 8 and 32 atoms end.

F_i takes g_ji from the slot of the reverse pair, so one wrong or missing slot changes two forces by the
size of a pair's gradient.  Doubles: 1e-10 of the largest force against the oracle; for the large cell, whose
tiles outnumber the grid, sum F = 0 to 1e-12 of sum |F| (3.4e6 pair terms, each of 1e-16 relative rounding).
"""

import numpy as np
import pytest
import torch

import oracle
from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _params(L, S):
    labels = synth.labels_from_level_table(levels.level_table(L))
    return synth.scaled_params(L, S, 6, 1.0, 5.0, labels, seed=L, radial_decay=0.5)


@pytest.mark.parametrize("sizes", [(1,), (1, 6), (8,), (9,), (31,), (32,), (33,), (24, 41), (1, 1, 62, 1), (130,)])
def test_forces_at_the_ends_of_tiles(gpu_lib, sizes):
    p = _params(6, 2)
    rng = np.random.default_rng(sum(sizes))
    cfgs = [synth.random_small_config(rng, n, n, species_pool=(0, 1), max_species=2) for n in sizes]
    # an atom that is its own neighbour through many images, and one without neighbours
    cfgs.append(synth.Config(np.array([[0.3, 2.0, -7.0]]), np.ones(1, dtype=np.int32), np.diag([2.3, 2.6, 3.1])))
    cfgs.append(synth.Config(np.array([[1.0, 2.0, 3.0]]), np.zeros(1, dtype=np.int32), np.diag([20.0, 20.0, 20.0])))
    b = synth.pack(cfgs)
    model = mtp.Model.from_params(p, "fp64")
    out = model.eval_batch(dev(b.pos), dev(b.types, torch.int32), dev(b.cells), dev(b.cfg_off, torch.int32))
    pot = oracle.Potential(p)
    ref = np.concatenate([pot.eval(c)["forces"] for c in cfgs])
    assert np.abs(out["forces"].cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max() + 1e-13


def test_more_tiles_than_blocks(gpu_lib):
    x, H = synth.supercell(synth.LATTICES["fcc"](), (27, 27, 27))
    rng = np.random.default_rng(3)
    order = rng.permutation(len(x))  # neighbours far apart in the numbering
    x = (x + rng.normal(0, 0.1, size=x.shape))[order]
    b = synth.pack([synth.Config(x, rng.integers(0, 2, size=len(x)).astype(np.int32), H)])
    model = mtp.Model.from_params(_params(4, 2), "fp64")
    F = model.eval_batch(dev(b.pos), dev(b.types, torch.int32), dev(b.cells), dev(b.cfg_off, torch.int32))["forces"]
    assert float(F.abs().max()) > 0
    assert float(F.sum(0).abs().max()) <= 1e-12 * float(F.abs().sum())
