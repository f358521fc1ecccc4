"""The integer unpacking of fp64 packed results against the fp64 equations it
replaces (eqs. 9-10, 13-14), compiled for the host: random magnitudes around
every digit position, exact ties of both roundings and their neighbours, zero,
subnormal and non-finite values, q over its range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1110_5765_gb300", "csrc")
SHIM = r"""
#include <cmath>
#include <cstring>
#include <cstdint>
#define __device__
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static inline long long __double_as_longlong(double d) { long long b; memcpy(&b, &d, 8); return b; }
static inline double __longlong_as_double(long long b) { double d; memcpy(&d, &b, 8); return d; }
static inline double __hiloint2double(int h, int l) {
    return __longlong_as_double((long long)(((uint64_t)(uint32_t)h << 32) | (uint32_t)l)); }
#include "tdg_digits.cuh"
extern "C" void sym(const double *r, int n, int q, double *out) {
    for (int i = 0; i < n; ++i)
        out[i] = q <= 31 ? tdg::sym_digit<true>(r[i], q) : tdg::sym_digit<false>(r[i], q); }
extern "C" void sym_wide(const double *r, int n, int q, double *out) {
    for (int i = 0; i < n; ++i) out[i] = tdg::sym_digit<false>(r[i], q); }
extern "C" void asym(const double *r, int n, int q, double *out) {
    for (int i = 0; i < n; ++i) {
        double d[4];
        tdg::asym_digits<4>(r[i], q, d);
        memcpy(out + 4 * i, d, 32); } }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("digits")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "digits.so"
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-fwrapv", "-I", CSRC, "-o", str(so),
                    str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(so))


def _call(fn, r, q, width):
    out = np.empty((r.size, width))
    p = ctypes.POINTER(ctypes.c_double)
    fn(r.ctypes.data_as(p), r.size, q, out.ctypes.data_as(p))
    return out


def _values(q):
    g = np.random.default_rng(q)
    v = [g.standard_normal(4000) * 2.0 ** g.integers(-80, 120, 4000)]
    Q = 2.0 ** q
    k = g.integers(-60, 60, 400).astype(float)
    for step in (0.5, Q / 2, Q, Q * Q / 2, 1 / Q, 0.5 / Q):         # ties of every rounding
        ties = k * step
        v += [ties, np.nextafter(ties, np.inf), np.nextafter(ties, -np.inf), ties + 0.5,
              ties - 0.5, ties + 0.25 * g.integers(-4, 5, 400)]
    big = g.integers(1, 1 << 50, 400).astype(float)
    v += [big + 0.5, -big - 0.5, np.array([0.0, -0.0, 5e-324, -1e-310, np.inf, -np.inf, np.nan,
                                           2.0 ** 52 + 0.5, 2.0 ** 53 + 2, -2.0 ** 63, 1e300])]
    return np.ascontiguousarray(np.concatenate(v))


def _same(a, b):
    return np.array_equal(a + 0.0, b + 0.0, equal_nan=True)


@pytest.mark.parametrize("q", [1, 6, 17, 21, 22, 30, 31, 32, 35, 44, 53, 60])
def test_symmetric_digit(host, q):
    r = _values(q)
    with np.errstate(all="ignore"):
        u = np.rint(r)
        t = np.rint(u * 2.0 ** -q)
        # fma(-Q, t, u): Q t and u are multiples of ulp(u) or Q, so u - Q t is exact
        ref = np.where(np.isfinite(r), u - t * 2.0 ** q, np.nan)
    assert _same(_call(host.sym, r, q, 1)[:, 0], ref)
    assert _same(_call(host.sym_wide, r, q, 1)[:, 0], ref)


@pytest.mark.parametrize("q", [6, 17, 21, 22, 31, 35, 44, 60])
def test_asymmetric_digits(host, q):
    r = _values(q)
    got = _call(host.asym, r, q, 4)
    x = r.copy()
    with np.errstate(all="ignore"):
        for d in range(4):
            ref = np.rint(x)
            assert _same(got[:, d], ref), d
            x = (x - ref) * 2.0 ** q
