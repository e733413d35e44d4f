"""What an MD run that fails leaves behind: the positions of the failing step, and both positions and
velocities as they came in where the first list already fails."""

import numpy as np
import pytest
import torch

from oracle import levels
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu

MASSES = [26.98, 58.69]
OVERFLOW = 4


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _setup(seed):
    cfg = synth.perturbed("fcc", (4, 4, 4), 0.05, np.random.default_rng(seed), n_species=2)
    p = synth.scaled_params(8, 2, 8, 1.0, 5.0, synth.labels_from_level_table(levels.level_table(8)), seed,
                            radial_decay=0.5)
    return cfg, p, synth.maxwell_velocities(cfg.types, MASSES, 300.0, seed)


def _run(p, cfg, precision, x, v, steps, cap, skin, dt=1.0):
    model = mtp.Model.from_params(p, precision)
    model.set_skin(skin)
    model.set_neighbor_capacity(cap)
    model.md_run(x, v, dev(cfg.types, torch.int32), dev(cfg.cell), MASSES, dt, steps)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_first_list_overflows(gpu_lib, precision):
    cfg, p, v0 = _setup(3)
    x, v = dev(cfg.pos), dev(v0)
    with pytest.raises(mtp.MTPError) as ei:
        _run(p, cfg, precision, x, v, 5, 20, 0.3)
    assert ei.value.code == OVERFLOW
    assert torch.equal(x, dev(cfg.pos)) and torch.equal(v, dev(v0))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_later_list_overflows(gpu_lib, precision):
    cfg, p, _ = _setup(4)
    # atoms drift towards the centre of the cell: the lists grow from rebuild to rebuild
    centre = 0.5 * cfg.cell.sum(axis=0)
    v0 = -0.01 * (cfg.pos - centre)
    small = mtp.Model.from_params(p, precision)
    counts = small.neighbors(dev(cfg.pos), dev(cfg.cell[None]), dev([0, cfg.n], torch.int32), 0.3)[0]
    cap = int(counts.max())
    for steps in range(1, 30):
        x, v = dev(cfg.pos), dev(v0)
        try:
            _run(p, cfg, precision, x, v, steps, cap, 0.3)
        except mtp.MTPError as e:
            assert e.code == OVERFLOW and steps > 1
            break
    else:
        pytest.fail("no list overflowed")
    failed = []
    for more in (steps, steps + 3):  # whether or not another step would have followed
        x, v = dev(cfg.pos), dev(v0)
        with pytest.raises(mtp.MTPError):
            _run(p, cfg, precision, x, v, more, cap, 0.3)
        failed.append(x)
    good = dev(cfg.pos)
    _run(p, cfg, precision, good, dev(v0), steps, 1024, 0.3)
    # (forces are sums in a fixed order: equal up to the last bits)
    for x in failed:
        assert (x - good).abs().max().item() <= 1e-10
