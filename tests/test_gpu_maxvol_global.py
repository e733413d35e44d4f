"""MaxVol of so many rows that the blocks' rows, and their positions, lie in global memory (Sec. 2.3), so that the
blocks' shares of B and of A overlap, and of tall, narrow matrices with more blocks than columns.  The selection equals a plain restatement (elimination with partial
pivoting, then swaps by C = B A^-1 from scratch); A A^-1 = 1 within 64 eps m cond(A)."""

import numpy as np
import pytest
import torch

from paper_2007_08555_gb300 import mtp

pytestmark = pytest.mark.gpu


def _maxvol(B):
    B = B / np.abs(B).max(axis=0)
    W, sel = B.copy(), []
    for k in range(B.shape[1]):
        p = int(np.argmax(np.abs(W[:, k])))
        sel.append(p)
        W[:, k + 1:] -= np.outer(W[:, k] / W[p, k], W[p, k + 1:])
        W[p] = 0.0
    swaps = 0
    while True:
        C = np.abs(B @ np.linalg.inv(B[sel]))
        k, j = divmod(int(np.argmax(C)), B.shape[1])
        if C[k, j] <= 1.001:
            return sel, swaps
        sel[j] = k
        swaps += 1


@pytest.mark.parametrize("n,m", [(20011, 29), (90001, 29), (120007, 32), (200003, 61), (33, 1), (517, 2),
                                 (1000, 9), (100003, 9), (3001, 17)])
def test_selection_from_many_rows(gpu_lib, n, m):
    model = mtp.Model(12, 2, 8, 2.0, 5.0)
    model.set_grade_kind(True, np.arange(m, dtype=np.int32))
    rng = np.random.default_rng(n + m)
    B = rng.normal(size=(n, m)) * 10.0 ** rng.uniform(-1, 1, size=m)
    rows, swaps, _ = model.select_active_set(torch.as_tensor(B, device="cuda"))
    sel, want = _maxvol(B)
    assert rows.cpu().tolist() == sel and swaps == want
    A, ai, _ = mtp.mtp_get_active_set(model.h, m)
    assert np.array_equal(A, B[sel])
    assert np.abs(A @ ai - np.eye(m)).max() <= 64 * np.finfo(float).eps * m * np.linalg.cond(A)
