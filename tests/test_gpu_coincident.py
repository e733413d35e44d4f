"""Two atoms at one place (r_ij = 0): energy, site energies and basis rows are finite (Eqs. 2-5 hold at r = 0;
only the gradient of |r| does not exist there) and equal the oracle's, at the tolerances of the evaluation
tests.  Levels on both sides of the double path's change of contraction."""

import numpy as np
import pytest
import torch

import oracle
from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
@pytest.mark.parametrize("L", [6, 16, 18])
def test_energy_of_coincident_atoms(gpu_lib, precision, tol, L):
    cfg = synth.perturbed("bcc", (2, 3, 2), 0.1, np.random.default_rng(L), n_species=2)
    cfg.pos[3] = cfg.pos[7]
    p = synth.scaled_params(L, 2, 8, 1.0, 5.0, synth.labels_from_level_table(levels.level_table(L)), seed=L,
                            radial_decay=0.5)
    ref = oracle.Potential(p).eval(cfg, want_b=True)
    out = mtp.Model.from_params(p, precision).eval_batch(dev(cfg.pos), dev(cfg.types, torch.int32), dev(cfg.cell[None]),
                                                         dev([0, cfg.n], torch.int32), site=True, b_atoms=True)
    site, b = out["site"].cpu().numpy(), out["b_atoms"].cpu().numpy()
    scale = np.abs(ref["site"]).max()
    assert abs(out["energy"].item() - ref["energy"]) <= tol * scale * cfg.n
    assert np.abs(site - ref["site"]).max() <= tol * scale
    assert (np.abs(b - ref["b_atoms"]) <= tol * np.abs(ref["b_atoms"]).max(axis=0)).all()
