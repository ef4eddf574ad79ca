"""A residual norm that becomes non-finite: the iteration's sweeps and update
leave the state and the increments as they were, the context (a single case)
or only its own case (a batch) fails, and the other case goes on as alone."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu

OPTS = [dict(), dict(scheme=1), dict(lusgs=1), dict(jvp=1), dict(precision=1)]


def _cloud():
    return cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))


def _huge(n, at):
    """A free stream with one point of speed of sound 1e80 and density 1e120: its mass flux squared overflows."""
    rho, u, v, p = np.full(n, 1.0), np.full(n, 0.6), np.zeros(n), np.full(n, 1.0 / 1.4)
    rho[at], p[at] = 1e120, 1e280
    return rho, u, v, p


@pytest.mark.parametrize("opts", OPTS)
def test_single_case(opts):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = _cloud()
    at = int(np.flatnonzero(np.asarray(cloud.flag) == 0)[100])
    s = lk.Solver(cloud, 0.6, 0.0, cfl=1.0, inner_iters=0, first_order_iters=100, **opts)
    s.run(3)
    s.set_state(*_huge(cloud.n, at))
    U, dU = s.field(lk.FIELD_U), s.field(lk.FIELD_DU)
    st, done = s.run(2, check=False)
    assert st == lk.ERR_DIVERGED
    assert np.array_equal(s.field(lk.FIELD_U), U)
    assert np.array_equal(s.field(lk.FIELD_DU), dU)
    assert not np.isfinite(s.residuals()[-1])


@pytest.mark.parametrize("opts", OPTS)
def test_one_case_of_a_batch(opts):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = _cloud()
    n = cloud.n
    at = int(np.flatnonzero(np.asarray(cloud.flag) == 0)[100])
    kw = dict(cfl=1.0, inner_iters=0, first_order_iters=100, **opts)
    solo = lk.Solver(cloud, 0.6, 0.0, **kw)
    b = lk.Solver.batch([cloud, cloud], [(0.6, 0.0), (0.6, 0.0)], **kw)
    good, bad = [np.full(n, 1.0), np.full(n, 0.6), np.zeros(n), np.full(n, 1.0 / 1.4)], _huge(n, at)
    solo.set_state(*good)
    b.set_state(*[np.concatenate([g, h]) for g, h in zip(good, bad)])
    U, dU = b.field(lk.FIELD_U), b.field(lk.FIELD_DU)
    solo.run(3)
    b.run(3, check=False)
    assert b.case_info(0)["status"] == lk.OK and b.case_info(0)["iters"] == 3
    assert b.case_info(1)["status"] == lk.ERR_DIVERGED and b.case_info(1)["iters"] == 1
    assert np.array_equal(b.field(lk.FIELD_U)[:n], solo.field(lk.FIELD_U))
    assert np.array_equal(b.field(lk.FIELD_U)[n:], U[n:])
    assert np.array_equal(b.field(lk.FIELD_DU)[n:], dU[n:])
