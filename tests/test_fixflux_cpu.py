"""The fixed-point split fluxes (csrc/lskum_fixflux.cuh) compiled for the host
against mpmath: every flux component within one FP64 rounding (2^-53) of the
sum of its terms' magnitudes, over the accepted ranges and at their edges
(slow and fast, hot and cold, thin and dense states, zero velocities,
interval edges of the tables); states outside are reported; the committed
table header is what the committed generator writes; the weighted sum keeps
the weights' and differences' bits."""
import ctypes
import importlib.util
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2406_07441_gb300", "csrc")

_SRC = r"""
#include <algorithm>
#include <cstdint>
using std::max;
#define __device__
#define __forceinline__ inline
#include "lskum_fluxtable.h"
#include "lskum_fixflux.cuh"
using namespace lskum;
extern "C" int flux_one(const double *z, int dir, int pos, double *hi, double *lo)
{
    const uint64_t *T = (const uint64_t *)kFluxTable;
    FxState s;
    FxFlux f;
    uint32_t bad = 0;
    fx_state(T, z[0], z[1], z[2], z[3], s, bad);
    if (dir == 0) fx_flux(T, s, s.u, s.su, s.v, s.sv, pos != 0, f, bad);
    else fx_flux(T, s, s.v, s.sv, s.u, s.su, pos != 0, f, bad);
    const int64_t g[4] = {(int64_t)f.rm, (int64_t)f.ga, (int64_t)f.go, (int64_t)f.g3};
    for (int c = 0; c < 4; c++) {  // an int64 as two doubles, exactly
        hi[c] = (double)(g[c] >> 32);
        lo[c] = (double)(uint32_t)g[c];
    }
    return bad >> 31;
}
extern "C" double weighted(const int *wh, const int *wl, const long long *gi, const long long *g0, int n)
{
    FxSum s = {};
    for (int k = 0; k < n; k++) fx_add(s, wh[k], wl[k], (uint64_t)gi[k], (uint64_t)g0[k]);
    return fx_total(s);
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
        L = ctypes.CDLL(so)
        L.weighted.restype = ctypes.c_double
        yield L


def _q(rho, u, v, p):
    b = rho / (2 * p)
    return np.array([np.log(rho) + 2.5 * np.log(b) - b * (u * u + v * v), 2 * b * u, 2 * b * v, -2 * b])


def _exact(z, d, pos):
    """The flux of the state with these (double) q-variables, and its terms' magnitudes."""
    z = [mp.mpf(float(t)) for t in z]
    b = -z[3] / 2
    u, v = z[1] / (2 * b), z[2] / (2 * b)
    rho = mp.exp(z[0] + b * (u * u + v * v)) * b ** mp.mpf(-2.5)
    p = rho / (2 * b)
    a, o = (v, u) if d else (u, v)
    sg = 1 if pos else -1
    S = a * mp.sqrt(b)
    A = mp.erfc(-sg * S) / 2
    B = mp.exp(-S * S) / (2 * mp.sqrt(mp.pi * b))
    m = rho * (a * A + sg * B)
    k = rho * (u * u + v * v) / 2
    G = [m, m * a + p * A, m * o, a * (3.5 * p + k) * A + sg * (3 * p + k) * B]
    ma = rho * (abs(a) + B)
    mag = [ma, ma * abs(a) + p, ma * abs(o), abs(a) * (3.5 * p + k) + (3 * p + k) * B]
    return G, mag


def _states():
    rng = np.random.default_rng(5)
    out = []
    for _ in range(120):  # subsonic to moderately supersonic flow about the free stream's entropy
        T = rng.uniform(0.3, 1.2)
        rho = (T * 1.4) ** 2.5 * rng.uniform(0.5, 1.0)
        c = np.sqrt(1.4 * T)
        m, th = rng.uniform(0, 2.0), rng.uniform(0, 2 * np.pi)
        out.append(_q(rho, m * c * np.cos(th), m * c * np.sin(th), rho * T))
    for T in (0.127, 0.5, 0.714, 0.998, 1.99):  # edges: temperatures, zero and tiny velocities, thin gas
        for u, v in ((0.0, 0.0), (1e-9, -1e-300), (-0.7, 0.0), (0.0, 1.1), (3.9 * T, -3.9 * T)):
            for rho in (1e-3, 0.2, 0.99 * (1.0 / (2 * T)) ** -2.5 * 0.99):
                out.append(_q(rho, u, v, rho * T))
    for j in (1, 17, 256, 400):  # S on and beside the intervals' edges
        for e in (-1, 0, 1):
            b = 0.7
            out.append(_q(0.9, (j / 256) / np.sqrt(b) * (1 + e * 2.0 ** -52), 0.1, 0.9 / (2 * b)))
    return out


def _call(L, z, d, pos):
    hi, lo = np.zeros(4), np.zeros(4)
    dp = ctypes.POINTER(ctypes.c_double)
    bad = L.flux_one(np.ascontiguousarray(z).ctypes.data_as(dp), d, pos, hi.ctypes.data_as(dp), lo.ctypes.data_as(dp))
    return bad, [mp.mpf(float(h)) * 2 ** 32 + mp.mpf(float(l)) for h, l in zip(hi, lo)]


def test_fluxes_within_one_fp64_rounding_of_their_terms(lib):
    accepted = 0
    with mp.workdps(40):
        for z in _states():
            for d in (0, 1):
                for pos in (0, 1):
                    bad, f = _call(lib, z, d, pos)
                    if bad:
                        continue
                    accepted += 1
                    G, mag = _exact(z, d, pos)
                    sg = 1 if pos else -1
                    for c, (s, unit) in enumerate(((sg, 59), (1, 57), (sg, 57), (sg, 55))):
                        err = abs(s * f[c] / mp.mpf(2) ** unit - G[c])
                        assert err <= mp.mpf(2) ** -53 * mag[c] + mp.mpf(4) / 2 ** unit, (z, d, pos, c, float(err))
    assert accepted > 600


@pytest.mark.parametrize("state", [
    (1.0, 6.0, 0.0, 0.7), (1.0, 0.0, -5.0, 0.7), (1.0, 0.1, 0.1, 2.5), (1.0, 0.1, 0.1, 0.06), (9.0, 0.1, 0.0, 2.0),
    (1e-9, 0.0, 0.0, 1e-9), (1.0, 2.9, 0.0, 0.4)])
def test_states_outside_the_ranges_are_reported(lib, state):
    assert any(_call(lib, _q(*state), d, 1)[0] for d in (0, 1))


def test_non_finite_and_unphysical_states_are_reported(lib):
    ok = _q(1.0, 0.5, 0.1, 0.7)
    for c in range(4):
        for v in (np.nan, np.inf, -np.inf, 1e300):
            z = ok.copy()
            z[c] = v
            assert _call(lib, z, 0, 1)[0], (c, v)
    z = ok.copy()
    z[3] = 0.3  # beta < 0
    assert _call(lib, z, 0, 1)[0]
    assert not _call(lib, ok, 0, 1)[0]


def test_weighted_sum_is_exact(lib):
    rng = np.random.default_rng(9)
    n = 510
    wh = rng.integers(-(2 ** 30) // n, 2 ** 30 // n, n).astype(np.int32)
    wl = rng.integers(-(2 ** 23), 2 ** 23 + 1, n).astype(np.int32)
    gi = rng.integers(-(2 ** 61), 2 ** 61, n)
    g0 = gi - rng.integers(-(2 ** 62), 2 ** 62, n)
    g0[:9] = gi[:9]
    got = lib.weighted(wh.ctypes.data_as(ctypes.c_void_p), wl.ctypes.data_as(ctypes.c_void_p),
                       gi.ctypes.data_as(ctypes.c_void_p), g0.ctypes.data_as(ctypes.c_void_p), n)
    ref = sum((mp.mpf(int(w)) + mp.mpf(int(l)) / 2 ** 24) * (int(a) - int(b))
              for w, l, a, b in zip(wh, wl, gi, g0)) / mp.mpf(2) ** 32
    # exact integers, five roundings of the total, and per term wl's product
    # with the difference's low word (2^-24 2^23 2^31 2^-32 at most)
    assert abs(got - ref) <= abs(ref) * 5 * 2 ** -53 + n * 0.25


def test_table_header_equals_the_generators_output():
    spec = importlib.util.spec_from_file_location("gen_fluxtable", os.path.join(CSRC, "gen_fluxtable.py"))
    gen = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(gen)
    with tempfile.TemporaryDirectory() as d:
        out = os.path.join(d, "t.h")
        gen.main(out)
        with open(out) as a, open(os.path.join(CSRC, "lskum_fluxtable.h")) as b:
            assert a.read() == b.read()
