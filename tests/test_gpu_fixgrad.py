"""The q-derivatives in fixed point on the device against extended precision:
first order and after inner iterations, every number of lanes per point, on a
jittered and on a stretched cloud, with and without states outside the
fixed-point ranges, against a bound that follows the roundings (of q, of the
weights, of each pass's result) through the passes."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud
from tests.test_gpu_fixflux import _state

pytestmark = pytest.mark.gpu

CLOUDS = {
    "jittered": lambda: cg.naca0012_jittered(48, 20),
    "o-grid": lambda: cg.naca0012_block(40, 16),
}


def _derivatives(cloud, q, K):
    """Extended-precision derivatives [2][n][4] of q [n][4], and a bound on the
    error of a computed form: 2^-57 of q, deg 2^-51 relative per product, 2^-57
    of the stencil's largest difference scale per pass."""
    f = np.longdouble
    off, idx = cloud.nbr_off, cloud.nbr_idx
    n = cloud.n
    own = np.repeat(np.arange(n), np.diff(off))
    deg = np.diff(off).astype(f)[:, None]
    dx, dy = (f(1) * cloud.x)[idx] - (f(1) * cloud.x)[own], (f(1) * cloud.y)[idx] - (f(1) * cloud.y)[own]

    def total(v):
        out = np.zeros((n,) + v.shape[1:], f)
        np.add.at(out, own, v)
        return out

    sxx, syy, sxy = total(dx * dx), total(dy * dy), total(dx * dy)
    det = sxx * syy - sxy * sxy
    w = [(syy[own] * dx - sxy[own] * dy) / det[own], (sxx[own] * dy - sxy[own] * dx) / det[own]]
    # weights in double carry the determinant's cancellation
    wrel = f(2) ** -50 * (sxx * syy / det)[:, None]
    sw = [total(np.abs(t))[:, None] for t in w]
    dq = (f(1) * q)[idx] - (f(1) * q)[own]
    size = np.zeros((n, 4), f)
    np.maximum.at(size, own, np.abs(dq))
    g = [total(t[:, None] * dq) for t in w]
    first = [t.copy() for t in g]
    unit = f(2) ** -57
    e0 = [s * (unit + (deg * f(2) ** -51 + wrel) * size) for s in sw]
    err = [t.copy() for t in e0]
    for _ in range(K):
        new, nerr = [], []
        for a in range(2):
            step = dx[:, None] * (g[0][idx] - g[0][own]) + dy[:, None] * (g[1][idx] - g[1][own])
            mag = (np.abs(dx)[:, None] * (np.abs(g[0][idx]) + np.abs(g[0][own])) +
                   np.abs(dy)[:, None] * (np.abs(g[1][idx]) + np.abs(g[1][own])))
            emag = (np.abs(dx)[:, None] * (err[0][idx] + err[0][own]) + np.abs(dy)[:, None] * (err[1][idx] + err[1][own]))
            aw = np.abs(w[a])[:, None]
            top = np.zeros((n, 4), f)  # a weight is rounded relative to the largest
            np.maximum.at(top, own, mag)
            new.append(first[a] - total(w[a][:, None] * step) / 2)
            nerr.append(e0[a] + total(aw * emag) / 2 + (deg * f(2) ** -50 + wrel) * sw[a] * top + unit * sw[a])
        g, err = new, nerr
    return g, err


@pytest.mark.parametrize("hard", [0.0, 0.05])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_derivatives_against_extended_precision(name, hard):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("fixgrad_" + name, CLOUDS[name])
    prim = _state(cloud, 0.63, 2.0, hard)
    for K in (0, 1, 2, 3):
        ref = None
        for tpp in (1, 2, 4, 8):
            s = lk.Solver(cloud, 0.63, 2.0, cfl=1.0, inner_iters=K, first_order_iters=1)
            s.set_launch_shape(tpp, 32)
            s.set_state(*prim)
            q = s.field(lk.FIELD_Q)
            s.run(1, check=False)
            got = [s.field(lk.FIELD_QX), s.field(lk.FIELD_QY)]
            if ref is None:
                ref, bound = _derivatives(cloud, q, K)
            for a in range(2):
                assert np.all(np.abs(got[a] - ref[a]) <= bound[a]), (K, tpp, a)
