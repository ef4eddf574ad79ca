"""The q-derivatives of cases with fast free streams, whose units are scaled
per case, against extended precision: the derivatives are linear, so each
component over its case's power of two obeys the bound of the slow cases."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud
from tests.test_gpu_fixgrad import _derivatives

pytestmark = pytest.mark.gpu


def _powers(mach):
    """Of the first and of the second and third components, as the library chooses them (aoa 0)."""
    q0, q1 = abs(2.5 * np.log(0.7) - 0.7 * mach ** 2), 1.4 * mach
    return max(0, int(np.ceil(np.log2(q0 / 6)))), max(0, int(np.ceil(np.log2(q1 / 3))))


@pytest.mark.parametrize("hard", [0.0, 0.05])
@pytest.mark.parametrize("mach", [2.5, 6.0, 40.0])
def test_derivatives_of_fast_free_streams(mach, hard):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("fixgrad_jittered", lambda: cg.naca0012_jittered(48, 20))
    rng = np.random.default_rng(51)
    n = cloud.n
    rho, p = rng.uniform(0.9, 1.1, n), rng.uniform(0.68, 0.75, n)
    u, v = mach * rng.uniform(0.95, 1.05, n), mach * rng.uniform(-0.1, 0.1, n)
    far = np.flatnonzero(rng.random(n) < hard)  # (out of the scaled range as well)
    u[far] *= 9.0
    s0, s1 = _powers(mach)
    scale = 2.0 ** -np.array([s0, s1, s1, 0.0])
    for K in (0, 2):
        for tpp in (1, 8):
            s = lk.Solver(cloud, mach, 0.0, cfl=0.1, inner_iters=K, first_order_iters=1)
            s.set_launch_shape(tpp, 32)
            s.set_state(rho, u, v, p)
            q = s.field(lk.FIELD_Q)
            s.run(1, check=False)
            ref, bound = _derivatives(cloud, q * scale, K)
            for a, f in enumerate((lk.FIELD_QX, lk.FIELD_QY)):
                assert np.all(np.abs(s.field(f) * scale - ref[a]) <= bound[a]), (K, tpp, a)


def test_a_batch_of_slow_and_fast_cases_equals_the_single_solves():
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20k", lambda: cg.naca0012_jittered(48, 20, kinetic_outer=True))
    conds = [(0.7, 1.0), (2.4, 0.0), (5.0, 2.0)]
    kw = dict(cfl=0.1, inner_iters=2, first_order_iters=100, farfield=lk.FARFIELD_KINETIC)
    b = lk.Solver.batch([cloud] * 3, conds, **kw)
    b.run(3)
    G = b.field(lk.FIELD_QX).reshape(3, cloud.n, 4)
    for c, (m, a) in enumerate(conds):
        s = lk.Solver(cloud, m, a, **kw)
        s.run(3)
        assert np.array_equal(s.field(lk.FIELD_QX), G[c]), c
