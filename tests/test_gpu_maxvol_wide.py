"""MaxVol at the widest active sets that the nonlinear criterion takes (Sec. 2.3): m + S^2 N_mu N_Q columns, 5580
at lev_max 20 with 8 species and 16 radial functions.  As many rows as columns: every row is selected, no
swap is made, and A A^-1 = 1 within 64 eps m cond(A)."""

import numpy as np
import pytest
import torch

from paper_2007_08555_gb300 import mtp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [5106, 5107, 5580])
def test_widest_active_sets(gpu_lib, width):
    model = mtp.Model(20, 8, 16, 1.0, 5.0)
    model.set_grade_kind(True, np.arange(width, dtype=np.int32))
    assert model.grade_width == width
    g = torch.Generator("cuda").manual_seed(width)
    # rows near a permuted, scaled identity: well conditioned, pivots off the diagonal
    perm = torch.randperm(width, generator=g, device="cuda")
    B = torch.randn((width, width), dtype=torch.float64, device="cuda", generator=g) * (0.1 / width ** 0.5)
    B[torch.arange(width, device="cuda"), perm] += 1.0
    rows, swaps, largest = model.select_active_set(B)
    assert sorted(rows.cpu().tolist()) == list(range(width)) and swaps == 0
    assert largest == pytest.approx(1.0, rel=1e-9)
    _, ai, _ = mtp.mtp_get_active_set(model.h, width)
    err = (B[rows.long()] @ torch.as_tensor(ai, device="cuda") - torch.eye(width, dtype=torch.float64, device="cuda"))
    assert err.abs().max().item() <= 64 * 2.0 ** -52 * width * 1.5
