"""Points outside the fixed-point ranges: the residual's FP64 form.  In mixed
precision its neighbour sums are compensated, as they are exact inside the
ranges: on long neighbour lists R then depends on how the lanes split them far
less than without."""
import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud
from tests.wide import two_rings

pytestmark = pytest.mark.gpu


def _hypersonic(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(0.8, 1.2, n), 6.0 + rng.uniform(-0.5, 0.5, n), rng.uniform(-0.5, 0.5, n),
            rng.uniform(0.6, 0.8, n))


def test_mixed_precision_compensates_the_sums_out_of_the_ranges():
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("wide_48x20", lambda: two_rings(cg.naca0012_jittered(48, 20)))
    spread = {}
    for precision in (0, 1):
        R = {}
        for tpp in (1, 2, 4):
            s = lk.Solver(cloud, 6.0, 0.0, cfl=0.1, inner_iters=0, first_order_iters=1, precision=precision)
            s.set_launch_shape(tpp, 4)
            s.set_state(*_hypersonic(cloud.n, 3))
            s.run(1, check=False)
            R[tpp] = s.field(lk.FIELD_R)
        spread[precision] = np.sqrt(sum(np.mean((R[t] - R[1]) ** 2, axis=0) for t in (2, 4)))
    # 80 to 170 additions of a running sum against the last rounding of each lane's
    assert np.all(spread[0] > 0)
    assert np.all(spread[1] < 0.5 * spread[0]), spread
