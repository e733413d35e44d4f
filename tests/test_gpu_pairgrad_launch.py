"""Evaluations on both sides of the rule that starts the pair gradients early or only after the contraction: between
half a wave and four blocks per SM in float from lev_max 16 on, in double by level and blocks.  The results do not
depend on it: the same atoms as part of a batch of another size give the same energies and forces."""

import numpy as np
import pytest
import torch

from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 2e-5)])
@pytest.mark.parametrize("L", [10, 12, 16])
def test_batches_of_every_launch(gpu_lib, precision, L, tol):
    p = synth.scaled_params(L, 2, 8, 1.0, 5.0, synth.labels_from_level_table(levels.level_table(L)), seed=L,
                            radial_decay=0.5)
    cfg = synth.perturbed("fcc", (4, 4, 4), 0.1, np.random.default_rng(L), n_species=2)  # 256 atoms, 16 blocks
    model = mtp.Model.from_params(p, precision)
    ref = None
    for copies in (1, 5, 9, 11, 37, 40):  # 16 to 640 blocks of eight lanes per atom
        b = synth.pack([cfg] * copies)
        args = (dev(b.pos), dev(b.types, torch.int32), dev(b.cells), dev(b.cfg_off, torch.int32))
        out = None
        for _ in range(3):  # eager, captured, replayed
            out = model.eval_batch(*args, out=out)
            e, F = out["energy"].cpu().numpy(), out["forces"].cpu().numpy().reshape(copies, -1)
            if ref is None:
                ref = (e[0], F[0])
            assert np.abs(e - ref[0]).max() <= tol * abs(ref[0])
            assert np.abs(F - ref[1]).max() <= tol * np.abs(ref[1]).max()
