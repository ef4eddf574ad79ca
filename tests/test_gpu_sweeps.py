"""The sweeps' launch: levels above and below the size where interior points
change from four lanes to two give the same bits (each case of a batch whose
joint levels are wide equals its single solve, whose levels are not)."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,jvp,lusgs,shape", [(0, 0, 0, (1, 32)), (1, 0, 0, (2, 4)), (0, 1, 0, (1, 32)),
                                                       (0, 0, 1, (2, 32))])
def test_wide_levels_of_a_batch_equal_the_single_solves_bit_for_bit(precision, jvp, lusgs, shape):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit336x136", lambda: cg.naca0012_jittered(336, 136))
    conds = [(0.6, 1.0), (0.7, -1.0)]
    kw = dict(cfl=1.0 if lusgs else 100.0, inner_iters=2, first_order_iters=10, precision=precision, jvp=jvp, lusgs=lusgs)
    b = lk.Solver.batch([cloud] * 2, conds, **kw)
    b.set_launch_shape(*shape)
    assert b.run(6) == 6
    U = b.field(lk.FIELD_U).reshape(2, cloud.n, 4)
    dU = b.field(lk.FIELD_DU).reshape(2, cloud.n, 4)
    for c, (m, a) in enumerate(conds):
        s = lk.Solver(cloud, m, a, **kw)
        s.set_launch_shape(*shape)
        assert s.run(6) == 6
        assert np.array_equal(s.field(lk.FIELD_U), U[c])
        assert np.array_equal(s.field(lk.FIELD_DU), dU[c])


@pytest.mark.parametrize("precision,lusgs", [(0, 0), (1, 0), (0, 1)])
def test_increment_products_of_a_zero_increment_are_zero(precision, lusgs):
    """The fluxes that the increment products subtract are formed apart from
    those at the incremented state: for a zero increment they agree bit for
    bit, so a uniform free stream (no wall in reach, residual 0) stays as it is."""
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))
    s = lk.Solver(cloud, 0.6, 0.0, cfl=10.0, inner_iters=0, first_order_iters=100, jvp=lk.JVP_INCREMENT,
                  precision=precision, lusgs=lusgs)
    s.run(1)  # the wall's residual reaches its neighbours' neighbours only
    R, dU = s.field(lk.FIELD_R), s.field(lk.FIELD_DU)
    U = s.field(lk.FIELD_U)
    far = np.hypot(np.asarray(cloud.x) - 0.5, np.asarray(cloud.y)) > 10.0
    assert np.all(R[far] == 0.0)
    quiet = far & np.all(dU == 0.0, axis=1)
    assert quiet.any()
    assert np.array_equal(U[quiet], np.broadcast_to(U[quiet][0], U[quiet].shape))
