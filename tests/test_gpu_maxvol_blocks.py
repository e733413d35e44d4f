"""MaxVol over several blocks at the sizes where the sharing of rows can go wrong (Sec. 2.3).

Widths of one to a few columns (one block), as many rows as columns, blocks without rows, rows that
exceed shared memory (kept in global memory), widths and row counts that no block count divides; ties
(duplicate rows) and a zero pivot.  Selection and swaps equal the oracle's; A^-1 lies within the forward
error of an inverse, 64 eps m cond(A D), of numpy's.
"""

import numpy as np
import pytest
import torch

from oracle import maxvol
from paper_2007_08555_gb300 import mtp

pytestmark = pytest.mark.gpu


def _rows(n, m, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=(n, m)) * 10.0 ** np.linspace(-3, 6, m)


def _select(B):
    n, m = B.shape
    sel = torch.full((m,), -1, dtype=torch.int32, device="cuda")
    ai = torch.zeros((m, m), dtype=torch.float64, device="cuda")
    swaps = mtp.mtp_select_active_set_noalloc(n, m, torch.as_tensor(B, device="cuda"), sel, ai)
    return sel.cpu().numpy(), swaps, ai.cpu().numpy()


@pytest.mark.parametrize("n,m", [(1, 1), (9, 1), (2, 2), (5, 3), (33, 4), (17, 17), (129, 61), (61, 61), (230, 229),
                                 (6000, 9), (40000, 3), (60000, 2)])
def test_selection_at_the_edges_of_the_blocks(gpu_lib, n, m):
    B = _rows(n, m, 7 * n + m)
    sel, swaps, ai = _select(B)
    sel_o, swaps_o, _ = maxvol.maxvol(B)
    assert sel.tolist() == sel_o.tolist() and swaps == swaps_o
    A_s, d = maxvol.equilibrate(B[sel_o])
    ref = d[:, None] * np.linalg.inv(A_s)
    tol = 64 * np.finfo(float).eps * m * np.linalg.cond(A_s)
    scaled = ai / d[:, None]  # the inverse of the equilibrated matrix
    assert np.abs(scaled - ref / d[:, None]).max() <= tol * np.linalg.norm(ref / d[:, None], 2)


@pytest.mark.parametrize("n,lev", [(920, 20), (60000, 8)])
def test_selection_with_a_model(gpu_lib, n, lev):
    model = mtp.Model(lev, 1, 4, 2.0, 5.0)
    B = _rows(n, model.m, n)
    sel, swaps, largest = model.select_active_set(torch.as_tensor(B, device="cuda"))
    sel_o, swaps_o, g_o = maxvol.maxvol(B)
    assert sel.cpu().tolist() == sel_o.tolist() and swaps == swaps_o
    assert largest == pytest.approx(g_o, rel=1e-9)


def test_ties_go_to_the_first_of_equal_rows(gpu_lib):
    B = _rows(40, 17, 3)
    B = np.concatenate([B, B, B[::-1]])
    sel, swaps, _ = _select(B)
    sel_o, swaps_o, _ = maxvol.maxvol(B)
    assert sel.tolist() == sel_o.tolist() and swaps == swaps_o


def test_rows_without_a_pivot_are_singular(gpu_lib):
    B = _rows(50, 9, 4)
    B[:, 5] = 0.0
    for bad in (B, np.where(np.arange(9) == 2, np.nan, _rows(50, 9, 4))):
        with pytest.raises(mtp.MTPError) as ei:
            _select(np.ascontiguousarray(bad))
        assert ei.value.code == 5


@pytest.mark.parametrize("lev", [2, 4, 6, 18])
def test_inverse_of_a_given_active_set(gpu_lib, lev):
    model = mtp.Model(lev, 1, 4, 2.0, 5.0)
    m = model.m
    A = np.random.default_rng(lev).normal(size=(m, m))
    mtp.mtp_set_active_set(model.h, A)
    _, ai, _ = mtp.mtp_get_active_set(model.h, m)
    ref = np.linalg.inv(A)
    tol = 64 * np.finfo(float).eps * m * np.linalg.cond(A)
    assert np.abs(ai - ref).max() <= tol * np.linalg.norm(ref, 2)
