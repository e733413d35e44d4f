"""A MaxVol launch that fails reports -1 and leaves no error behind for the next call's cudaGetLastError: the
compiled launchers (the object of the library) against a fake of the CUDA runtime whose calls fail in turn."""

import ctypes
import os
import subprocess

import pytest

from paper_2007_08555_gb300 import build

FAKE = r"""
#include <cstddef>
struct CUstream_st;
static int pending = 0, fail_at = -1, calls = 0;
static int step() { return calls++ == fail_at ? (pending = 720) : 0; }
extern "C" {
int cudaGetLastError() { int e = pending; pending = 0; return e; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return 0; }
int cudaMemcpyAsync(void*, const void*, size_t, int, CUstream_st*) { return 0; }
int cudaStreamSynchronize(CUstream_st*) { return 0; }
int cudaMemsetAsync(void*, int, size_t, CUstream_st*) { return step(); }
int cudaFuncSetAttribute(const void*, int, int) { return step(); }
int cudaLaunchCooperativeKernel(const void*, ...) { return step(); }
int __cudaGetKernel(void**, const void*) { return 0; }
int __cudaLaunchKernel(...) { return 0; }
unsigned __cudaPushCallConfiguration(...) { return 0; }
int __cudaPopCallConfiguration(...) { return 0; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(...) {}
void __cudaRegisterVar(...) {}
}
namespace mtp {
int launch_maxvol(int, int, const double*, double*, double*, size_t, int*, int*, double*, double*, double, int, int*, int*,
                  double*, CUstream_st*, int);
int launch_invert(int, const double*, double*, double*, int*, CUstream_st*);
}
extern "C" int run(int invert, int n, int m, int fail, int* left) {
  static double none[4];
  int zero = 0;
  fail_at = fail;
  calls = pending = 0;
  int r = invert ? mtp::launch_invert(m, none, none, none, &zero, nullptr)
                 : mtp::launch_maxvol(n, m, none, none, none, 1 << 20, &zero, &zero, none, none, 1e-3, 100, &zero, &zero, none,
                                      nullptr, 0);
  *left = pending;
  return r;
}
"""


@pytest.fixture(scope="module")
def launchers(tmp_path_factory):
    obj = os.path.join(build.OUT, "mtp_maxvol.o")
    if not os.path.exists(obj):
        build.build()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.cpp").write_text(FAKE)
    subprocess.run(["g++", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", str(d / "fake.so"), str(d / "fake.cpp"), obj], check=True)
    return ctypes.CDLL(str(d / "fake.so"))


@pytest.mark.parametrize("invert", [0, 1])
@pytest.mark.parametrize("n,m,steps", [(9, 3, 2), (232, 116, 4)])  # one block; several: two memsets come first
def test_a_failed_launch_leaves_no_error(launchers, invert, n, m, steps):
    left = ctypes.c_int()
    for fail in range(steps + 1):  # the last one lets every call pass
        assert launchers.run(invert, n, m, fail, ctypes.byref(left)) == (1 if fail == steps else -1)
        assert left.value == 0, fail
