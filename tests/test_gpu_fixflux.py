"""The fixed-point residual on the device: points with states outside its
ranges (hypersonic, cold, hot, dense) take the FP64 form and agree with the
oracle beside points that do not, for every number of lanes per point; inside
the ranges R does not depend on that number (exact sums)."""
import numpy as np
import pytest

import oracle as O
from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu


def _state(cloud, mach, aoa, hard):
    rng = np.random.default_rng(31)
    n = cloud.n
    al = np.deg2rad(aoa)
    rho, p = rng.uniform(0.8, 1.1, n), rng.uniform(0.65, 0.8, n)
    u, v = mach * np.cos(al) + rng.uniform(-0.1, 0.1, n), mach * np.sin(al) + rng.uniform(-0.1, 0.1, n)
    k = np.flatnonzero(rng.random(n) < hard)
    rho[k], p[k] = 10.0 ** rng.uniform(-2, 1, k.size), 10.0 ** rng.uniform(-1.5, 1, k.size)
    u[k], v[k] = rng.uniform(-6, 6, k.size), rng.uniform(-6, 6, k.size)
    return rho, u, v, p


@pytest.mark.parametrize("hard", [0.0, 0.02, 0.5])
def test_residual_in_and_out_of_the_fixed_point_ranges(hard):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))
    o = O.Oracle(cloud)
    prim = _state(cloud, 0.63, 2.0, hard)
    ref, first = None, None
    for tpp in (1, 2, 4, 8):
        s = lk.Solver(cloud, 0.63, 2.0, cfl=1.0, inner_iters=0, first_order_iters=1)
        s.set_launch_shape(tpp, 32)
        s.set_state(*prim)
        U = s.field(lk.FIELD_U)
        s.run(1, check=False)
        R = s.field(lk.FIELD_R)
        if ref is None:
            ref = o.run(U, 1, cfl=1.0, K=0, first_order=1)["R"]
            first = R
        assert np.max(np.abs(R - ref)) <= 1e-10 * np.max(np.abs(ref)), tpp
        if hard == 0.0:
            assert np.array_equal(R, first), tpp  # the same integer sums
