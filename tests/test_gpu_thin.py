"""Thin gas on the device: the residual of a state with density and pressure
scaled by a power of two is that residual scaled, up to the rounding of the
first q-variable, which shifts by the power's logarithm."""
import numpy as np
import pytest

import oracle as O
from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tpp", [1, 8])
@pytest.mark.parametrize("power", [4, 10, 18])
def test_residual_scales_with_the_density(power, tpp):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))
    rng = np.random.default_rng(41)
    n = cloud.n
    rho, p = rng.uniform(0.7, 1.2, n), rng.uniform(0.6, 0.8, n)
    u, v = 0.6 + rng.uniform(-0.1, 0.1, n), rng.uniform(-0.1, 0.1, n)
    R, U = {}, {}
    for k in (0, power):
        s = lk.Solver(cloud, 0.63, 2.0, cfl=1.0, inner_iters=0, first_order_iters=1)
        s.set_launch_shape(tpp, 32)
        s.set_state(rho * 2.0 ** -k, u, v, p * 2.0 ** -k)
        U[k] = s.field(lk.FIELD_U)
        s.run(1, check=False)
        R[k] = s.field(lk.FIELD_R)
    assert np.array_equal(U[power] * 2.0 ** power, U[0])
    # what relative errors of the points' densities of up to d do to R: the
    # first q-variable (|q1| < 2 + power ln 2) carries 1.5 units in its last
    # place (logarithm 1, sum 1/2), at the scaled and at the unscaled state, and
    # the fluxes and weights add two roundings
    def units(x):
        return 1.5 * 2.0 ** (np.floor(np.log2(x)) - 52)
    d = units(2 + power * np.log(2)) + units(1.9) + 2 * 2.0 ** -53
    o = O.Oracle(cloud)
    eps = 2.0 ** -30
    sign = rng.choice([-1.0, 1.0], (n, 1))
    a, b = (o.run(x, 1, cfl=1.0, K=0, first_order=1)["R"] for x in (U[0], U[0] * (1 + eps * sign)))
    for c in range(4):
        dev = R[power][:, c] * 2.0 ** power - R[0][:, c]
        assert np.sqrt(np.mean(dev ** 2)) <= d * np.sqrt(np.mean((b[:, c] - a[:, c]) ** 2)) / eps, c
