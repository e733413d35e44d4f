"""MaxVol where rounding decides (Sec. 2.3): matrices of small integers are full of ties, and ranks are lost exactly
or not by the last bit.  The selection is defined by the elimination, the inverse, C and the swaps in double
precision in this order of operations, which no number of blocks may change: a host restatement with the
same operations must select the same rows, make the same swaps and find the same matrices singular."""

import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2007_08555_gb300 import mtp

pytestmark = pytest.mark.gpu

RESTATEMENT = r"""
#include <cmath>
#include <vector>
#include <utility>
using V = std::vector<double>;
// returns the swaps, or -1: singular, -2: limit of swaps
extern "C" int maxvol(int n, int m, const double* raw, int* sel) {
  V B(raw, raw + (size_t)n * m), W;
  for (int c = 0; c < m; ++c) {
    double mx = 0;
    for (int r = 0; r < n; ++r) mx = fmax(mx, fabs(raw[(size_t)r * m + c]));
    if (!(mx > 0)) return -1;
    const double d = 1.0 / mx;
    for (int r = 0; r < n; ++r) B[(size_t)r * m + c] *= d;
  }
  W = B;
  std::vector<int> perm(n);
  for (int r = 0; r < n; ++r) perm[r] = r;
  for (int k = 0; k < m; ++k) {
    int p = k;
    for (int r = k; r < n; ++r)
      if (fabs(W[(size_t)perm[r] * m + k]) > fabs(W[(size_t)perm[p] * m + k])) p = r;
    std::swap(perm[k], perm[p]);
    const double* pk = &W[(size_t)perm[k] * m];
    if (pk[k] == 0) return -1;
    for (int r = k + 1; r < n; ++r) {
      double* w = &W[(size_t)perm[r] * m];
      const double l = w[k] / pk[k];
      for (int c = k + 1; c < m; ++c) w[c] = std::fma(-l, pk[c], w[c]);
    }
    sel[k] = perm[k];
  }
  auto inverse = [&](V& A) {  // Gauss-Jordan with row interchanges on [A | 1]
    const int w = 2 * m;
    V G((size_t)m * w, 0.0);
    for (int r = 0; r < m; ++r) {
      for (int c = 0; c < m; ++c) G[(size_t)r * w + c] = B[(size_t)sel[r] * m + c];
      G[(size_t)r * w + m + r] = 1.0;
    }
    for (int k = 0; k < m; ++k) {
      int p = k;
      for (int r = k; r < m; ++r)
        if (fabs(G[(size_t)r * w + k]) > fabs(G[(size_t)p * w + k])) p = r;
      if (G[(size_t)p * w + k] == 0) return false;
      for (int c = 0; c < w; ++c) std::swap(G[(size_t)k * w + c], G[(size_t)p * w + c]);
      const double inv = 1.0 / G[(size_t)k * w + k];
      for (int c = 0; c < w; ++c) G[(size_t)k * w + c] *= inv;
      for (int r = 0; r < m; ++r) {
        const double f = G[(size_t)r * w + k];
        if (r != k)
          for (int c = 0; c < w; ++c) G[(size_t)r * w + c] = c == k ? 0.0 : std::fma(-f, G[(size_t)k * w + c], G[(size_t)r * w + c]);
      }
    }
    A.resize((size_t)m * m);
    for (int r = 0; r < m; ++r)
      for (int c = 0; c < m; ++c) A[(size_t)r * m + c] = G[(size_t)r * w + m + c];
    return true;
  };
  V Ai, C((size_t)n * m), row(m), col(n);
  if (!inverse(Ai)) return -1;
  for (int r = 0; r < n; ++r)
    for (int c = 0; c < m; ++c) {
      double s = 0;
      for (int k = 0; k < m; ++k) s = std::fma(B[(size_t)r * m + k], Ai[(size_t)k * m + c], s);
      C[(size_t)r * m + c] = s;
    }
  for (int swaps = 0;; ++swaps) {
    size_t at = 0;
    for (size_t e = 0; e < C.size(); ++e)
      if (fabs(C[e]) > fabs(C[at])) at = e;
    if (fabs(C[at]) <= 1.0 + 1e-3) return inverse(Ai) ? swaps : -1;
    if (swaps == 100 * m) return -2;
    const int k = (int)(at / m), j = (int)(at % m);
    const double ckj = C[at];
    for (int c = 0; c < m; ++c) row[c] = C[(size_t)k * m + c] - (c == j ? 1.0 : 0.0);
    for (int r = 0; r < n; ++r) col[r] = C[(size_t)r * m + j];
    for (int r = 0; r < n; ++r)
      for (int c = 0; c < m; ++c) C[(size_t)r * m + c] -= col[r] * row[c] / ckj;
    sel[j] = k;
  }
}
"""


@pytest.fixture(scope="module")
def restated(tmp_path_factory):
    d = tmp_path_factory.mktemp("maxvol")
    (d / "m.cpp").write_text(RESTATEMENT)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "m.so"), str(d / "m.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "m.so"))

    def run(B):
        sel = np.full(B.shape[1], -1, dtype=np.int32)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        return lib.maxvol(B.shape[0], B.shape[1], p(B), p(sel)), sel.tolist()

    return run


def _compare(restated, kind, seed):
    rng = np.random.default_rng([seed, len(kind)])
    m = int(rng.integers(2, 80))
    n = int(m + rng.integers(0, 2 * m + 1))
    lo, hi = {"signs": (-2, 3), "bits": (0, 2), "wide": (-50, 51), "rank_lost": (-5, 6)}[kind]
    B = rng.integers(lo, hi, size=(n, m)).astype(np.float64)
    if kind == "rank_lost":  # (in exact arithmetic; the last pivot is zero or a rounding error)
        B[:, -1] = 3 * B[:, 0] - 7 * B[:, (m - 1) // 2]
    want, rows = restated(B)
    sel = torch.full((m,), -1, dtype=torch.int32, device="cuda")
    try:
        got = mtp.mtp_select_active_set_noalloc(n, m, torch.as_tensor(B, device="cuda"), sel)
    except mtp.MTPError as e:
        got = {5: -1, 6: -2}[e.code]
    assert got == want
    if want >= 0:
        assert sel.cpu().tolist() == rows


@pytest.mark.parametrize("kind", ["signs", "bits", "wide", "rank_lost"])
@pytest.mark.parametrize("seed", range(40))
def test_selection_of_integer_matrices(gpu_lib, restated, kind, seed):
    _compare(restated, kind, seed)


@pytest.mark.parametrize("seed", [68, 4675, 5032])
def test_swaps_that_the_last_bit_decides(gpu_lib, restated, seed):
    _compare(restated, "bits", seed)
