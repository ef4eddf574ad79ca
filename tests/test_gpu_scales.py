"""States scaled by extreme powers of two (density and pressure alike: the
equations are linear in the scale): what is representable runs as the unscaled
state does."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu


def _run(power, **opts):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))
    rng = np.random.default_rng(61)
    n = cloud.n
    rho, p = rng.uniform(0.95, 1.05, n), rng.uniform(0.69, 0.73, n)
    u, v = 0.6 + rng.uniform(-0.02, 0.02, n), rng.uniform(-0.02, 0.02, n)
    s = lk.Solver(cloud, 0.6, 0.0, cfl=1.0, inner_iters=1, first_order_iters=100, **opts)
    s.set_state(rho * 2.0 ** power, u, v, p * 2.0 ** power)
    assert s.run(2) == 2
    return s.field(lk.FIELD_U) * 2.0 ** -power, s.residuals()


# The first q-variable of the scaled state, up to 512 ln 2 = 355, is rounded to
# 2^-45; two iterations at CFL 1 pass on a few times that (the unscaled
# states' densities, of order one, move by their own order in the outer cells).
TOL = 64 * 2.0 ** -45


@pytest.mark.parametrize("opts", [dict(), dict(scheme=1), dict(lusgs=1), dict(jvp=1)])
def test_a_dense_state_whose_norm_is_finite_does_not_diverge(opts):
    ref, _ = _run(0, **opts)
    U, hist = _run(480, **opts)
    assert np.all(np.isfinite(hist)) and hist[0] > 1e140
    assert np.max(np.abs(U - ref)) <= TOL


@pytest.mark.parametrize("opts", [dict(jvp=1), dict(jvp=1, lusgs=1), dict()])
@pytest.mark.parametrize("power", [-520, -500])
def test_a_state_of_which_products_underflow(power, opts):
    """(The norm's squares underflow too: only the state is compared.)"""
    ref, _ = _run(0, **opts)
    U, _ = _run(power, **opts)
    assert np.max(np.abs(U - ref)) <= TOL
