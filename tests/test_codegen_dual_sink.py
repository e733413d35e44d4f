"""dL/dxi of a tile of 32 atoms as the loss gradient's generated tangent contraction sums it (Sec. 2.2), on the
host in single precision: the sum over the atoms of ek v - t is a double sum of the float values and
tangents (34 roundings: a product, a difference and 32 additions), and lanes without an atom, whose moments
are NaN or infinite here, add nothing."""

import ctypes
import subprocess

import numpy as np
import pytest

from paper_2007_08555_gb300 import codegen


def _build(L, parts, tmp_path):
    prog = codegen.build_program(L)
    src = ["#include <cstddef>", "#define __device__", "#define __forceinline__ inline", "namespace gen {"]
    src += codegen.emit_dual_parts(prog, parts) + ["}"]
    src.append("""
struct Record {  // values and tangents as the sink gets them
  float *v, *t;
  void put(int, int al, float a, float b) { v[al] = a; t[al] = b; }
};
extern "C" void tile(int parts, int C, int n, const float* m, const float* mt, const float* xi, const double* ek,
                     int M, float* v, float* t, double* dxt) {
  static float adj[gen::NDSLOT * 32], adt[gen::NDSLOT * 32];
  static double s[gen::MAXDALPHA * 33];
  int alpha[gen::MAXDALPHA];
  for (int g = 0; g < parts; ++g) {
    int na = 0;
    for (int l = 0; l < 32; ++l) {
      gen::DxiSink sink{l < n ? ek[l] : 0.0, l < n, s, alpha, l};
      na = gen::dual_part(g, m + l, mt + l, adj + l, adt + l, xi, sink);
      Record rec{v + (size_t)l * M, t + (size_t)l * M};
      gen::dual_part(g, m + l, mt + l, adj + l, adt + l, xi, rec);
    }
    gen::DxiSink any{0.0, false, s, alpha, 0};
    for (int q = 0; q < na; ++q) dxt[alpha[q]] = any.sum(q);
  }
}""")
    cpp, so = tmp_path / "tile.cpp", tmp_path / "tile.so"
    cpp.write_text("\n".join(src) + "\n")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(so), str(cpp)], check=True)
    return prog, ctypes.CDLL(str(so))


@pytest.mark.parametrize("L,parts", [(8, 1), (12, 2), (16, 4)])
@pytest.mark.parametrize("n", [1, 31, 32])
def test_tile_sum_is_a_double_sum_over_its_atoms(L, parts, n, tmp_path):
    prog, lib = _build(L, parts, tmp_path)
    rng = np.random.default_rng(100 * L + n)
    C, M = len(prog.comp_list), prog.basis.m
    m, mt = rng.normal(size=(2, C, 32)).astype(np.float32)
    m[:, n:] = np.where(rng.integers(0, 2, size=(C, 32 - n)) > 0, np.nan, np.inf)
    mt[:, n:] = -np.inf
    xi = rng.normal(size=M).astype(np.float32)
    ek = rng.normal(size=32) * 1e6  # large beside the tangents, of both signs: the sums cancel
    v, t = np.zeros((2, 32, M), dtype=np.float32)
    dxt = np.full(M, np.nan)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.tile(parts, C, n, p(m), p(mt), p(xi), p(ek), M, p(v), p(t), p(dxt))
    v, t = v[:n].astype(np.longdouble), t[:n].astype(np.longdouble)
    terms = ek[:n, None].astype(np.longdouble) * v - t
    bound = 34 * 2.0 ** -53 * (np.abs(ek[:n, None] * v) + np.abs(t)).sum(axis=0)
    assert (np.abs(dxt - terms.sum(axis=0)) <= bound).all()
