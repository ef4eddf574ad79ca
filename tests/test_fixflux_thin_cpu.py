"""Thin gas in the fixed-point split fluxes (csrc/lskum_fixflux.cuh compiled
for the host): with the scaling that the point's own state gives, an accepted
state's error is bounded relative to its terms' magnitudes alone, at every
density, and so is that of a neighbour some times thinner or denser than the
point whose scaling it takes; what overflows the scaling is reported."""
import ctypes
import os
import shutil
import struct
import subprocess
import tempfile

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

from tests.test_fixflux_cpu import CSRC, _exact, _q  # noqa: E402

_SRC = r"""
#include <algorithm>
#include <cstdint>
using std::max;
#define __device__
#define __forceinline__ inline
#include "lskum_fluxtable.h"
#include "lskum_fixflux.cuh"
using namespace lskum;
extern "C" int shift(unsigned rho, unsigned isb) { return (int)fx_shift(rho, isb); }
extern "C" int flux_one(const double *z, int sh, int dir, int pos, double *hi, double *lo)
{
    const uint64_t *T = (const uint64_t *)kFluxTable;
    FxState s;
    FxFlux f;
    uint32_t bad = 0;
    fx_state(T, z[0], z[1], z[2], z[3], s, bad, (uint32_t)sh);
    if (dir == 0) fx_flux(T, s, s.u, s.su, s.v, s.sv, pos != 0, f, bad);
    else fx_flux(T, s, s.v, s.sv, s.u, s.su, pos != 0, f, bad);
    const int64_t g[4] = {(int64_t)f.rm, (int64_t)f.ga, (int64_t)f.go, (int64_t)f.g3};
    for (int c = 0; c < 4; c++) {  // an int64 as two doubles, exactly
        hi[c] = (double)(g[c] >> 32);
        lo[c] = (double)(uint32_t)g[c];
    }
    return bad >> 31;
}
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
        yield ctypes.CDLL(so)


def _hi(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0] >> 32


def _shift(L, rho, T):
    return L.shift(_hi(rho), _hi(np.sqrt(2 * T)))


def _errors(L, z, sh, scale_z):
    """Largest error of an accepted state's components over both axes and halves, in units of 2^-53 of the
    magnitudes of the terms (of the state scale_z); None if a flux is reported."""
    dp = ctypes.POINTER(ctypes.c_double)
    worst = 0.0
    for d in (0, 1):
        for pos in (0, 1):
            hi, lo = np.zeros(4), np.zeros(4)
            if L.flux_one(np.ascontiguousarray(z).ctypes.data_as(dp), sh, d, pos, hi.ctypes.data_as(dp),
                          lo.ctypes.data_as(dp)):
                return None
            G, _ = _exact(z, d, pos)
            mag = _exact(scale_z, d, pos)[1]
            mag[2] = max(mag[1], mag[2])  # (the momentum across adds to the one along the other axis)
            for c, (s, unit) in enumerate(((2 * pos - 1, 59), (1, 57), (2 * pos - 1, 57), (2 * pos - 1, 55))):
                f = mp.mpf(float(hi[c])) * 2 ** 32 + mp.mpf(float(lo[c]))
                worst = max(worst, float(abs(s * f / mp.mpf(2) ** (unit + sh) - G[c]) / mag[c] * 2 ** 53))
    return worst


# Four units of the components (2^-59, 2^-57, 2^-57, 2^-55) at the least scaled
# rho/sqrt(beta) of 0.5 and T > 0.25: the energy's terms are at least 0.28 x
# 0.5 x 0.75, so 10 x 2^-53; 3 for the state's own (rho/sqrt(beta) in 2^-56 at
# the least 1/8), and one rounding of the terms.
BAR = 14.0


def test_error_relative_to_the_terms_at_every_density(lib):
    rng = np.random.default_rng(17)
    accepted = 0
    with mp.workdps(40):
        for lg in np.linspace(-6.0, 0.3, 64):
            for _ in range(3):
                rho, T = 10.0 ** lg * rng.uniform(0.8, 1.2), rng.uniform(0.27, 1.5)
                c, th = np.sqrt(1.4 * T) * rng.uniform(0, 2.0), rng.uniform(0, 2 * np.pi)
                z = _q(rho, c * np.cos(th), c * np.sin(th), rho * T)
                e = _errors(lib, z, _shift(lib, rho, T), z)
                if e is not None:
                    accepted += 1
                    assert e <= BAR, (rho, T, e)
    assert accepted > 120


@pytest.mark.parametrize("ratio", [0.05, 0.3, 1.9, 3.0, 40.0])
def test_a_neighbour_of_another_density(lib, ratio):
    """Its error counts against the denser of the two states; denser than the scaling holds it is reported."""
    rng = np.random.default_rng(18)
    taken = 0
    with mp.workdps(40):
        for lg in np.linspace(-5.0, -0.5, 16):
            rho, T = 10.0 ** lg, rng.uniform(0.5, 0.9)
            z0, z = _q(rho, 0.4, -0.2, rho * T), _q(rho * ratio, 0.3, 0.1, rho * ratio * T)
            e = _errors(lib, z, _shift(lib, rho, T), z if ratio > 1 else z0)
            taken += e is not None
            assert e is None or e <= BAR, (rho, T, e)
    assert taken == 0 if ratio > 10 else taken > 0


def test_the_scaling(lib):
    """A mantissa 1 + m taken for 2^m is short by at most 0.0861 in log2, two by 0.1722: at least 1/2, below 2^0.1722."""
    for T in (0.26, 0.714, 1.9):
        for rho in 10.0 ** np.linspace(-8, 1, 200):
            sh = _shift(lib, rho, T)
            rs = rho * np.sqrt(2 * T) * 2.0 ** sh
            top = 2.0 ** 0.1722
            assert (sh == 0 and rs >= 0.5) or (sh == 24 and rs < top) or 0.5 <= rs < top, (rho, T, sh)
