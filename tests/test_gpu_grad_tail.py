"""Loss gradient of atom counts that leave the last tile of 32 partly empty (Sec. 2.2).

The lanes without an atom work on whatever an earlier call left in their places.  A first batch whose
moments overflow (finite, but huge radial coefficients) leaves infinities and NaN there; a second, smaller
batch on the same model must give the gradient that a model without a history gives.  Both runs do the same
sums in the same order up to atomic additions: 1e-9 (double) and 1e-5 (float) of the largest entry.
"""

import numpy as np
import pytest
import torch

from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _args(sizes, S, seed):
    rng = np.random.default_rng(seed)
    b = synth.pack([synth.random_small_config(rng, n, n, species_pool=tuple(range(S)), max_species=S) for n in sizes])
    refs = (rng.normal(size=b.n_cfg), rng.normal(size=(b.n_atoms, 3)), rng.normal(size=(b.n_cfg, 9)))
    return (dev(b.pos), dev(b.types, torch.int32), dev(b.cells), dev(b.cfg_off, torch.int32), *map(dev, refs))


@pytest.mark.parametrize("precision,huge,tol", [("fp64", 1e307, 1e-9), ("fp32", 1e37, 1e-5)])
@pytest.mark.parametrize("L", [8, 16, 20])
@pytest.mark.parametrize("n", [1, 31, 40])
def test_gradient_after_a_batch_that_overflowed(gpu_lib, precision, huge, tol, L, n):
    p = synth.scaled_params(L, 2, 8, 1.0, 5.0, synth.labels_from_level_table(levels.level_table(L)), seed=L,
                            radial_decay=0.5)
    small = _args([n], 2, 5 * L + n)
    fresh = [t.cpu().numpy() for t in mtp.Model.from_params(p, precision).param_grad(*small)]
    model = mtp.Model.from_params(p, precision)
    model.set_params(c=np.full_like(p.c, huge))
    before = model.param_grad(*_args([40, 24], 2, L))
    assert not torch.isfinite(before[1]).all()
    model.set_params(c=p.c)
    for got, want in zip(model.param_grad(*small), fresh):
        got = got.cpu().numpy()
        assert np.isfinite(want).all() and np.isfinite(got).all()
        assert np.abs(got - want).max() <= tol * np.abs(want).max()
