"""The nested Horner adjoint (codegen.emit_horner), compiled for the host: the value of the polynomial of
df-weighted coefficients and the gradient of the f-weighted one equal the sums over components that they
stand for, for every level's set of monomials.  No GPU."""

import ctypes
import shutil
import subprocess

import numpy as np
import pytest

from paper_2007_08555_gb300 import codegen

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


@pytest.mark.parametrize("L", [4, 8, 10, 16, 20])
def test_horner_is_the_polynomials_gradient_and_value(L, tmp_path):
    prog = codegen.build_program(L)
    C = len(prog.comp_list)
    lines = codegen.emit_horner(prog, list(range(C + 1)))
    src = ["#define __device__", "#define __forceinline__ inline", "#define __restrict__", "namespace gen {"] + lines + ["}"]
    src.append('extern "C" void grad(double x, double y, double z, const double* f, const double* df, const double* adj, '
               "double* out) {")
    src.append("  gen::HornerF::grad<double>(x, y, z, f, df, adj, out[0], out[1], out[2], out[3]);")
    src.append("}")
    src.append('extern "C" void shared(const double* sl, double* dst, int sub) {')
    src.append("  gen::HornerF::adj_to_shared<double, 2, 1>(sl, dst, sub);")
    src.append("}")
    cpp, so = tmp_path / "h.cpp", tmp_path / "h.so"
    cpp.write_text("\n".join(src) + "\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", str(so), str(cpp)], check=True)
    lib = ctypes.CDLL(str(so))
    p = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    lib.grad.argtypes = [ctypes.c_double] * 3 + [ctypes.POINTER(ctypes.c_double)] * 4
    rng = np.random.default_rng(L)
    nmu = max(mu for mu, _ in prog.comp_list) + 1
    f, df, adj = rng.normal(size=nmu), rng.normal(size=nmu), rng.normal(size=C)
    v = rng.normal(size=3)
    # adj_to_shared: the components (one slot each here) in Horner's order, whichever lane writes them
    slots, dst = np.zeros(C * 32), np.full((C + 3) // 4 * 4, np.nan)
    slots[::32] = adj
    for sub in (0, 1):
        lib.shared(p(slots), p(dst), sub)
    assert dst[:C].tolist() == adj[codegen.horner_order(prog)].tolist()
    out = np.zeros(4)
    lib.grad(*v, p(f), p(df), p(dst), p(out))
    want, size = np.zeros(4), np.zeros(4)
    for t, (mu, m) in enumerate(prog.comp_list):
        mono = np.prod(v ** np.array(m))
        terms = [df[mu] * adj[t] * mono]
        for d in range(3):
            e = np.array(m)
            e[d] -= 1
            terms.append(f[mu] * adj[t] * m[d] * np.prod(v ** np.maximum(e, 0)) if m[d] else 0.0)
        want += terms
        size += np.abs(terms)
    np.testing.assert_array_less(np.abs(out - want), 1e-13 * size + 1e-300)
