"""Neighbour lists where the list kernel's staging changes form, bit-exact against the oracle's search.

One bin seen through many images (thin, flat and strongly sheared cells), few bins shared by many blocks,
dense cells whose candidates do not fit in one staging, atoms far outside their cell, and a large search
radius (a skin).
"""

import numpy as np
import pytest
import torch

import oracle
from paper_2007_08555_gb300 import mtp, synth

pytestmark = pytest.mark.gpu


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def _cells():
    rng = np.random.default_rng(5)
    out = {}
    for name, H in {"thin": np.diag([2.1, 14.0, 30.0]), "flat": np.diag([24.0, 19.0, 2.6]),
                    "sheared": np.array([[7.0, 0, 0], [6.0, 5.0, 0], [-5.5, 4.0, 8.0]]),
                    "two_bins": np.diag([10.4, 9.9, 9.9])}.items():
        n = max(1, int(abs(np.linalg.det(H)) * 0.05))
        out[name] = (rng.uniform(size=(n, 3)) @ H, H)
    H = np.diag([9.8, 9.8, 9.8])
    out["dense"] = (rng.uniform(size=(230, 3)) @ H, H)  # 2,000 candidates around one bin
    x, H = out["sheared"]
    out["wrapped"] = (x + rng.integers(-40, 41, size=x.shape) @ H, H)
    x, H = synth.supercell(synth.LATTICES["fcc"](), (3, 4, 11))
    out["bar"] = (x + rng.normal(0, 0.1, size=x.shape), H)
    return out


CELLS = _cells()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("names,skin", [((n,), 0.0) for n in CELLS] + [(("bar", "flat"), 1.5),
                                                                       (tuple(CELLS) * 3, 0.0)])
def test_lists_equal_the_oracle(gpu_lib, precision, names, skin):
    b = synth.pack([synth.Config(CELLS[n][0], np.zeros(len(CELLS[n][0]), dtype=np.int32), CELLS[n][1]) for n in names])
    model = mtp.Model(4, 1, 4, 1.0, 5.0, precision=precision)
    model.set_neighbor_capacity(512)
    counts, j, s, r = (t.cpu().numpy() for t in model.neighbors(dev(b.pos), dev(b.cells), dev(b.cfg_off, torch.int32),
                                                                skin))
    at = 0
    for k in range(b.n_cfg):
        c_o, j_o, s_o, r_o = oracle.neighbors(b.config(k).pos, b.config(k).cell, 5.0 + skin)
        m = int(np.sum(c_o))
        lo, hi = int(b.cfg_off[k]), int(b.cfg_off[k + 1])
        assert counts[lo:hi].tolist() == np.asarray(c_o).tolist()
        assert (j[at:at + m] - lo).tolist() == np.asarray(j_o).tolist()
        np.testing.assert_array_equal(s[at:at + m], np.asarray(s_o).reshape(-1, 3))
        np.testing.assert_array_equal(r[at:at + m], np.asarray(r_o).reshape(-1, 3))
        at += m
    assert at == len(j)
