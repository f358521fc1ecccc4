"""The statistics' arrival counters (CPU: the planner's header compiled for the host).

Two calls whose arrivals interleave on one plan, with the second call's coming in
while the first one's last warp is at work, must leave every counter at zero, so
that the next call decides its plan at its own last arrival, and not before."""
import ctypes
import os
import random
import subprocess

import pytest

from paper_1110_5765_gb300 import build

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
#include <vector>
#include <cuda.h>
#include <cuda_runtime.h>
using std::min; using std::max;
static struct { unsigned x; } lane_id;
#define threadIdx lane_id
static std::vector<int> *pending;       // slabs of the arrivals that come in meanwhile
static void meanwhile();
template <typename T> T __ldcg(const T *p) { meanwhile(); return *p; }
template <typename T> T __shfl_sync(unsigned, T v, int) { return v; }
template <typename T> T __shfl_xor_sync(unsigned, T v, int) { return v; }
static void __syncwarp() {}
static double __dmul_rn(double a, double b) { return a * b; }
static double __dadd_rn(double a, double b) { return a + b; }
static double __ddiv_rn(double a, double b) { return a / b; }
static double __dsqrt_rn(double a) { return std::sqrt(a); }
static int atomicExch(int *p, int v) { int o = *p; *p = v; return o; }
static int atomicCAS(int *p, int c, int v) { int o = *p; if (o == c) *p = v; return o; }
static size_t __cvta_generic_to_shared(const void *p) { return (size_t)p; }
static int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
#include "tdg_planner.cuh"

using namespace tdg;
static SlabFinish fin_of(int nM, int nK, int nN, int form, bool reuse, std::vector<double> &buf,
                         unsigned *counters) {
    SlabFinish f{};
    f.pp.form = form; f.pp.mode = MODE_TARGET; f.pp.L = 64; f.pp.p = 24;
    f.pp.nM = nM; f.pp.nK = nK; f.pp.nN = nN;
    f.mA = f.vA = f.mB = f.vB = buf.data();
    f.agg = buf.data() + 4096;
    set_slab_counters(f, counters, reuse);
    return f;
}
static SlabFinish *other;
static DevPlan *plan_rec;
static void meanwhile() {
    if (!pending || pending->empty()) return;
    std::vector<int> now;
    std::swap(now, *pending);
    for (int l : now) slab_finish(*other, l, plan_rec);
}
// arrivals first[0..n1) of one call; after `at` of them, and inside whatever its last
// warp of a slab does, those of a second call come in; then a call by itself.
// Returns 1 if that one decides its plan with its last arrival and no other, and every
// counter is zero before and after.
extern "C" int run(int nM, int nK, int nN, int reuse2, const int *first, int n1, const int *second,
                   int n2, int at, const int *third, int n3) {
    std::vector<double> buf(8192, 1.0);
    std::vector<unsigned> cnt(slab_count_bytes(nK) / sizeof(unsigned), 0u);
    DevPlan plan{};
    SlabFinish f1 = fin_of(nM, nK, nN, TDG_SYM, false, buf, cnt.data());
    SlabFinish f2 = fin_of(nM, nK, nN, TDG_SYM, reuse2 != 0, buf, cnt.data());
    plan_rec = &plan; other = &f2;
    std::vector<int> later(second, second + n2);
    for (int i = 0; i < n1; ++i) {
        if (i == at) pending = &later;
        slab_finish(f1, first[i], &plan);
    }
    meanwhile();
    for (int l : later) slab_finish(f2, l, &plan);
    pending = nullptr;
    for (unsigned c : cnt) if (c) return 0;
    plan.trho = -1.0;
    for (int i = 0; i < n3; ++i) {
        if (plan.trho != -1.0) return 0;
        slab_finish(f1, third[i], &plan);
    }
    if (plan.trho == -1.0) return 0;
    for (unsigned c : cnt) if (c) return 0;
    return 1;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("counters")
    (d / "shim.cpp").write_text(SHIM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    so = d / "counters.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-shared", "-fPIC", "-I", build.CSRC, "-I",
                    build.INCLUDE, "-I", cuda, "-o", str(so), str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("reuse", [0, 1])
@pytest.mark.parametrize("nM,nK,nN", [(1, 1, 1), (2, 3, 1), (3, 2, 4)])
def test_overlapping_calls_leave_the_counters_at_zero(host, nM, nK, nN, reuse):
    rng = random.Random(100 * nM + 10 * nK + nN + reuse)
    full = [k for k in range(nK) for _ in range(nM + nN)]
    part = [k for k in range(nK) for _ in range(nM)]

    def arr(v):
        return (ctypes.c_int * len(v))(*v)

    for _ in range(200):
        a, b, c = full[:], (part if reuse else full)[:], full[:]
        for v in (a, b, c):
            rng.shuffle(v)
        assert host.run(nM, nK, nN, reuse, arr(a), len(a), arr(b), len(b),
                        rng.randrange(len(a)), arr(c), len(c))
