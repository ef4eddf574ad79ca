"""The fixed-point q-derivative sums (csrc/lskum_fixgrad.cuh) compiled for the
host against Python integers: the sums are exact up to their limits, the value
is the exact sum to the nearest unit (and the bits cut off below it), out of
range is reported, and q converts to the nearest unit or to the mark."""
import ctypes
import os
import shutil
import subprocess
import tempfile
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2406_07441_gb300", "csrc")

_SRC = r"""
#define __device__
#define __forceinline__ inline
#include "lskum_fixgrad.cuh"
using namespace lskum;
extern "C" int grad_sum(const int *wh, const int *wl, const long long *d, int n, int b, int p, long long *v)
{
    GradSum s = {};
    for (int k = 0; k < n; k++) {
        int32_t h, l;
        if (k & 1) split_g(d[k], h, l);
        else split_word((uint64_t)d[k] + 0x80000000ull, h, l);
        if (join_g(h, l) != d[k]) return -1;
        grad_add(s, wh[k], wl[k], h, l);
    }
    int64_t r;
    const bool ok = grad_value(s.hh, grad_low(s, b), b, p, r);
    *v = r;
    return ok;
}
extern "C" long long fixed_q(double q, int c) { return fix_q(q, c); }
"""


@pytest.fixture(scope="module")
def lib():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    with tempfile.TemporaryDirectory() as d:
        src, so = os.path.join(d, "h.cpp"), os.path.join(d, "libh.so")
        with open(src, "w") as f:
            f.write(_SRC)
        subprocess.check_call([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so])
        L = ctypes.CDLL(so)
        L.fixed_q.restype = ctypes.c_longlong
        L.fixed_q.argtypes = [ctypes.c_double, ctypes.c_int]
        yield L


@pytest.mark.parametrize("n,b,p,top", [(20, 28, 0, 2 ** 63 - 2 ** 33), (40, 27, 3, 2 ** 62 - 1), (255, 23, 0, 2 ** 63 - 2 ** 33),
                                       (512, 22, 10, 2 ** 62 - 1), (2, 28, 0, 2 ** 40), (30, 20, 10, 2 ** 20)])
@pytest.mark.parametrize("edge", [False, True])
def test_sum_is_exact(lib, n, b, p, top, edge):
    rng = np.random.default_rng(n + b + p + edge)
    for _ in range(200):
        f = rng.random(n)
        wh = np.floor(f / f.sum() * (2 ** 31 - n - 1)).astype(np.int64)  # sum |wh| just below 2^31
        wl = rng.integers(-(2 ** (b - 1)), 2 ** (b - 1) + 1, n)
        while np.abs(wl).sum() >= 2 ** 31:
            wl //= 2
        if edge:  # every product of one sign, every difference at its limit
            d = np.array([top - int(rng.integers(0, 3)) for _ in range(n)], dtype=np.int64)
            wl = np.abs(wl)
        else:
            d = (rng.uniform(-1, 1, n) * float(top) * 0.999).astype(np.int64)
            wh *= rng.choice([-1, 1], n)
        v = ctypes.c_longlong()
        ok = lib.grad_sum(np.ascontiguousarray(wh, np.int32).ctypes.data_as(ctypes.c_void_p),
                          np.ascontiguousarray(wl, np.int32).ctypes.data_as(ctypes.c_void_p),
                          d.ctypes.data_as(ctypes.c_void_p), n, b, p, ctypes.byref(v))
        assert ok >= 0
        exact = sum(Fraction(int(w)) * int(t) + Fraction(int(x) * int(t), 2 ** b) for w, x, t in zip(wh, wl, d))
        exact = exact * Fraction(2) ** (p - 31)
        if ok:
            assert abs(Fraction(v.value) - exact) <= Fraction(1, 2) + Fraction(2) ** (p - b + 3)
        else:
            assert abs(exact) >= 2 ** 60
        if abs(exact) < 2 ** 60:
            assert ok


def test_q_in_units(lib):
    rng = np.random.default_rng(5)
    for c, unit, top in ((0, 59, 8.0), (1, 60, 4.0), (2, 60, 4.0), (3, 60, 4.0)):
        z = np.concatenate([rng.uniform(-top, top, 2000), 10.0 ** rng.uniform(-30, 0, 500), [0.0, -0.0, 2.0 ** -61, -(2.0 ** -1060)]])
        for x in z:
            v = lib.fixed_q(float(x), c)
            if v == -(2 ** 63):
                assert abs(x) >= top * (1 - 2.0 ** -20)
            else:
                assert abs(Fraction(v) - Fraction(float(x)) * 2 ** unit) <= Fraction(1, 2)
                assert abs(v) < 2 ** 62
        for x in (top, -top, 1e300, float("inf"), float("-inf"), float("nan")):
            assert lib.fixed_q(float(x), c) == -(2 ** 63)
