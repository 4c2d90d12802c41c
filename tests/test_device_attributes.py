"""Kernel attributes (shared memory above 48 KB) belong to a device: each
preparation of the FP64 form sets its own again for every device a process
uses, and not on every call.  Runs the library's own object files on the host
against a stand-in for the CUDA runtime that counts the calls per device."""
import ctypes
import os
import subprocess

import pytest

from paper_1504_00992_gb300 import build as BLD

STUB = r"""
#include <stddef.h>
int device = 0, calls[4], fail = 0;
int cudaGetDevice(int* d) { *d = device; return 0; }
int cudaFuncSetAttribute(const void* f, int a, int v) { if (fail) return 98; ++calls[device]; return 0; }
int cudaGetLastError(void) { return 0; }
void** __cudaRegisterFatBinary(void* p) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) {}
void __cudaUnregisterFatBinary(void** h) {}
void __cudaRegisterFunction(void** h, const char* f, char* d, const char* n, int t, void* a, void* b, void* c, void* e,
                            int* w) {}
void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int e, size_t s, int c, int g) {}
int __cudaGetKernel(void** k, const void* f) { *k = NULL; return 0; }
"""


@pytest.fixture(scope="module")
def prepared(tmp_path_factory):
    BLD.build()
    objs = [os.path.join(BLD.BUILDDIR, n + ".o") for n in ("qr_small", "jacobi_pre", "cholqr", "oz_proj",
                                                             "tebd_kernels")]
    if not all(os.path.exists(o) for o in objs):
        BLD.build(force=True)
    d = tmp_path_factory.mktemp("stub")
    src, stub, lib = str(d / "rt.c"), str(d / "rt.o"), str(d / "libprepare.so")
    with open(src, "w") as f:
        f.write(STUB)
    subprocess.run(["gcc", "-c", "-fPIC", "-o", stub, src], check=True)
    # symbolic: bound to the stand-in, whatever runtime the process has loaded; what it lacks is never called
    subprocess.run(["g++", "-shared", "-Wl,-z,lazy", "-Wl,-Bsymbolic", "-o", lib, stub, *objs], check=True)
    return ctypes.CDLL(lib, mode=os.RTLD_LAZY)


@pytest.mark.parametrize("name", ["_ZN2tg16qr_small_prepareEv", "_ZN2tg15jac_pre_prepareEv", "_ZN2tg14cholqr_prepareEv",
                                  "_ZN2tg10oz_prepareEv", "_ZN2tg13theta_prepareEv"])
def test_every_device_gets_its_attributes_once(prepared, name):
    dev, fail = ctypes.c_int.in_dll(prepared, "device"), ctypes.c_int.in_dll(prepared, "fail")
    calls = (ctypes.c_int * 4).in_dll(prepared, "calls")
    prepare = getattr(prepared, name)
    fail.value, dev.value = 1, 3
    assert prepare() != 0  # a failure is reported, and tried again
    fail.value = 0
    seen = []
    for d in (0, 1, 0, 1, 3):
        dev.value = d
        before = calls[d]
        assert prepare() == 0
        seen.append(calls[d] - before)
    assert seen[0] > 0 and seen[1] > 0 and seen[4] > 0
    assert seen[2] == 0 and seen[3] == 0
