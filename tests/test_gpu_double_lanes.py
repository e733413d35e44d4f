"""The double kernels at every number of lanes per atom against the oracle (1e-10 relative).

Slices of the moments over the warps of a block, contraction in parts (up to lev_max 16) and by the packed
program (above), pair gradients with every slice in shared memory (four lanes and more) and slice by slice;
atom counts around a tile of 32, atoms without neighbours, and the basis rows' sums.
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


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("L,S,NQ,sizes", [(2, 1, 4, (5,)), (10, 2, 8, (1, 31, 2)), (16, 3, 8, (33, 8, 20)),
                                          (18, 2, 6, (12, 21)), (20, 1, 8, (7,))])
def test_evaluation_at_every_lane_count(gpu_lib, L, S, NQ, sizes, lanes):
    labels = synth.labels_from_level_table(levels.level_table(L))
    p = synth.scaled_params(L, S, NQ, 1.0, 5.0, labels, seed=L, radial_decay=0.5)
    rng = np.random.default_rng(100 * L + lanes)
    cfgs = [synth.random_small_config(rng, n, n, species_pool=tuple(range(S)), max_species=S) for n in sizes]
    cfgs.append(synth.Config(np.array([[1.0, 2.0, 3.0]]), np.zeros(1, dtype=np.int32), np.diag([20.0, 20.0, 20.0])))
    b = synth.pack(cfgs)
    model = mtp.Model.from_params(p, "fp64")
    model.set_threads_per_atom(lanes, lanes)
    out = model.eval_batch(dev(b.pos), dev(b.types, torch.int32), dev(b.cells), dev(b.cfg_off, torch.int32), site=True,
                           b_rows=True)
    out = {k: v.cpu().numpy() for k, v in out.items()}
    pot = oracle.Potential(p)
    refs = [pot.eval(c, want_b=True) for c in cfgs]
    # a one-atom cell's forces cancel, so errors are taken against the batch's largest entry
    biggest = {key: max(np.abs(r[key]).max() for r in refs) for key in ("site", "forces", "virial", "b_atoms")}
    for k, (c, r) in enumerate(zip(cfgs, refs)):
        i = slice(int(b.cfg_off[k]), int(b.cfg_off[k + 1]))
        assert abs(out["energy"][k] - r["energy"]) <= 1e-10 * c.n * biggest["site"]
        assert np.abs(out["site"][i] - r["site"]).max() <= 1e-10 * biggest["site"]
        assert np.abs(out["forces"][i] - r["forces"]).max() <= 1e-10 * biggest["forces"]
        assert np.abs(out["virial"][k] - r["virial"]).max() <= 1e-10 * biggest["virial"]
        assert np.abs(out["b_rows"][k] - r["b_atoms"].sum(0)).max() <= 1e-10 * c.n * biggest["b_atoms"]
