"""The kernels' shared-memory attribute (CPU: the header compiled against a stand-in
runtime): set once on each device, and tried again after a failure."""
import ctypes
import subprocess

from paper_1110_5765_gb300 import build

RUNTIME = r"""
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 999 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
extern int g_device, g_fail, g_sets;
inline cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
template <typename K> cudaError_t cudaFuncSetAttribute(K, cudaFuncAttribute, int) {
    ++g_sets;
    return g_fail ? cudaErrorUnknown : cudaSuccess;
}
"""
SHIM = r"""
#include "tdg_optin.h"
int g_device, g_fail, g_sets;
static void kernel() {}
extern "C" int launch(int device, int fail, int *sets) {
    static tdg::SmemOptIn ok;
    g_device = device; g_fail = fail; g_sets = 0;
    int e = ok.allow(kernel, 232448);
    *sets = g_sets;
    return e;
}
"""


def test_once_per_device_and_again_after_a_failure(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "shim.cpp").write_text(SHIM)
    so = tmp_path / "optin.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", str(tmp_path), "-I", build.CSRC,
                    "-o", str(so), str(tmp_path / "shim.cpp")], check=True)
    lib, sets = ctypes.CDLL(str(so)), ctypes.c_int()

    def launch(device, fail=0):
        return lib.launch(device, fail, ctypes.byref(sets)), sets.value

    assert launch(0, fail=1) == (999, 1)
    assert launch(0) == (0, 1)
    assert launch(0, fail=1) == (0, 0)
    assert launch(3) == (0, 1)
    assert launch(3) == (0, 0) and launch(0) == (0, 0)
    assert launch(70) == (0, 1) and launch(70) == (0, 1)
