"""The bounded wait of the sweeps' launch runs out (one block never arrives;
every block returns after its limit): the call reports it, the state is that
of the last complete iteration, the increments are those of a new state, the
iteration and its norm are not counted, and the context goes on as one that
was given that state."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu

KW = dict(cfl=4.0, inner_iters=1, first_order_iters=4, cfl_ramp_iters=8.0)
OPTS = [dict(), dict(precision=1), dict(lusgs=1), dict(jvp=1), dict(lusgs=1, precision=1)]


def _cloud():
    return cached_cloud("block_80x32", lambda: cg.naca0012_block(80, 32))


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("lanes", [4, 32])
def test_a_timeout_leaves_the_last_state(opts, lanes):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = _cloud()
    s, t = (lk.Solver(cloud, 0.63, 2.0, **KW, **opts) for _ in range(2))
    for x in (s, t):
        x.set_launch_shape(2, lanes)
        assert x.run(3) == 3
    U, hist = s.field(lk.FIELD_U), s.residuals()
    s.set_wait_test(1, 1e-3)
    assert s.run(2, check=False) == (lk.ERR_TIMEOUT, 0)
    assert np.array_equal(s.field(lk.FIELD_U), U)
    assert not s.field(lk.FIELD_DU).any()
    assert np.array_equal(s.residuals(), hist)
    with pytest.raises(lk.LskumError) as e:
        s.time_phases(2)
    assert e.value.status == lk.ERR_TIMEOUT
    assert np.array_equal(s.field(lk.FIELD_U), U)
    assert not s.field(lk.FIELD_DU).any()
    assert np.array_equal(s.residuals(), hist)
    s.set_wait_test(0)
    t.set_conserved(U)
    assert s.run(4) == 4 and t.run(4) == 4
    assert np.array_equal(s.residuals(), t.residuals())
    for f in (lk.FIELD_U, lk.FIELD_DU):
        assert np.array_equal(s.field(f), t.field(f))


def test_a_timeout_of_a_batch():
    from paper_2406_07441_gb300 import lskum as lk
    cloud = _cloud()
    conds = [(0.63, 2.0), (0.4, 0.0)]
    s, t = (lk.Solver.batch([cloud] * 2, conds, **KW) for _ in range(2))
    for x in (s, t):
        assert x.run(3) == 3
    U, hist = s.field(lk.FIELD_U), [s.case_residuals(c) for c in range(2)]
    s.set_wait_test(1, 1e-3)
    assert s.run(2, check=False) == (lk.ERR_TIMEOUT, 0)
    assert np.array_equal(s.field(lk.FIELD_U), U)
    for c in range(2):
        assert s.case_info(c)["status"] == lk.OK and s.case_info(c)["iters"] == 3
        assert np.array_equal(s.case_residuals(c), hist[c])
    s.set_wait_test(0)
    t.set_conserved(U)
    assert s.run(4) == 4 and t.run(4) == 4
    assert np.array_equal(s.field(lk.FIELD_U), t.field(lk.FIELD_U))


def test_bad_arguments():
    from paper_2406_07441_gb300 import lskum as lk
    s = lk.Solver(_cloud(), 0.63, 2.0, **KW)
    for skip, limit in ((2, 1.0), (0, 0.0), (1, 11.0)):
        with pytest.raises(lk.LskumError) as e:
            s.set_wait_test(skip, limit)
        assert e.value.status == lk.ERR_ARG
    assert s.run(2) == 2
