"""dL/dc of batches with so many sums per warp that few warps fit on an SM, which then get longer chunks of atoms
(8 species, 16 radial functions): the loss is a sum over configurations, so a large batch must give the sum of
the smaller ones, whose chunks are short.  Tolerances as for the other sums of batches: 1e-10 of the
largest entry in double, 1e-5 in float."""

import numpy as np
import pytest
import torch

from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


@pytest.mark.parametrize("precision,L,n_cfg,tol", [("fp64", 6, 700, 1e-10), ("fp32", 20, 500, 1e-5), ("fp32", 10, 1000, 1e-5)])
def test_long_chunks(gpu_lib, precision, L, n_cfg, tol):
    S, NQ = 8, 16
    p = synth.scaled_params(L, S, NQ, 1.0, 5.0, synth.labels_from_level_table(levels.level_table(L)), seed=L,
                            radial_decay=0.5)
    rng = np.random.default_rng(n_cfg)
    cfgs = [synth.random_small_config(rng, 61, 83) for _ in range(n_cfg)]
    for c in cfgs:
        c.types = rng.integers(0, S, size=c.n).astype(np.int32)
    b = synth.pack(cfgs)
    refs = (rng.normal(size=b.n_cfg), rng.normal(size=(b.n_atoms, 3)), rng.normal(size=(b.n_cfg, 9)))
    model = mtp.Model.from_params(p, precision)

    def grad(lo, hi):
        q = synth.pack(cfgs[lo:hi])
        i0, i1 = int(b.cfg_off[lo]), int(b.cfg_off[hi])
        return [t.cpu().numpy() for t in model.param_grad(
            dev(q.pos), dev(q.types, torch.int32), dev(q.cells), dev(q.cfg_off, torch.int32), dev(refs[0][lo:hi]),
            dev(refs[1][i0:i1]), dev(refs[2][lo:hi]), (1.0, 0.01, 0.001))]

    whole, parts = grad(0, n_cfg), [0.0, 0.0, 0.0]
    for lo in range(0, n_cfg, 100):
        parts = [x + y for x, y in zip(parts, grad(lo, min(n_cfg, lo + 100)))]
    for x, y in zip(whole, parts):
        assert np.abs(x - y).max() <= tol * np.abs(y).max()
