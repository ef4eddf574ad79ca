"""The q-derivatives' units (csrc/lskum_fixgrad.cuh compiled for the host):
every free stream lies well inside the range that its case's powers of two
give, to within half a unit that is below FP64's own unit in the last place,
and low free streams keep the units 2^-59 and 2^-60."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from tests.test_fixgrad_cpu import CSRC

_SRC = r"""
#include <cstring>
#include "lskum_fixgrad.cuh"
using namespace lskum;
extern "C" int shift(const double *q) { return fix_shift(q); }
extern "C" int unit(int c, int s) { return fix_unit(c, s); }
extern "C" long long fixed_q(double q, int c, int s) { return fix_q(q, c, s); }
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
        L.fixed_q.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.c_int]
        yield L


MARK = -2 ** 63


@pytest.mark.parametrize("aoa", [0.0, 3.0, 45.0, -90.0])
@pytest.mark.parametrize("mach", [0.01, 0.85, 1.3, 2.1, 2.2, 2.86, 3.5, 6.0, 10.0, 40.0, 1000.0])
def test_free_streams_are_represented(lib, mach, aoa):
    u, v = mach * np.cos(np.deg2rad(aoa)), mach * np.sin(np.deg2rad(aoa))
    q = np.array([2.5 * np.log(0.7) - 0.7 * mach ** 2, 1.4 * u, 1.4 * v, -1.4])
    s = lib.shift(q.ctypes.data_as(ctypes.c_void_p))
    if mach <= 2.1:
        assert s == 0
    for c in range(4):
        unit = lib.unit(c, s)
        assert unit == 60 - (c == 0) or (c < 3 and np.spacing(max(abs(q[1]), abs(q[2]), abs(q[0]) / 8)) > 2.0 ** -unit)
        for near in (q[c], 1.3 * q[c]):
            got = lib.fixed_q(near, c, s)
            assert got != MARK and abs(got * 2.0 ** -unit - near) <= 2.0 ** -(unit + 1) + np.spacing(abs(near))
        # and the ends of the range are marked
        top = (8.0 if c == 0 else 4.0) * 2.0 ** ((59 if c == 0 else 60) - unit)
        assert lib.fixed_q(top, c, s) == MARK and lib.fixed_q(-np.inf, c, s) == MARK
        assert lib.fixed_q(top * (1 - 2.0 ** -20), c, s) != MARK
