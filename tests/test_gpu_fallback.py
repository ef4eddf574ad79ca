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


def _density_response(o, U, rng):
    """rms response of R's components to relative density errors of one unit (random signs)."""
    eps = 2.0 ** -30
    a, b = (o.run(x, 1, cfl=0.1, K=0, first_order=1)["R"]
            for x in (U, U * (1 + eps * rng.choice([-1.0, 1.0], (len(U), 1)))))
    return a, np.sqrt(np.mean((b - a) ** 2, axis=0)) / eps


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tpp", [1, 2, 4, 8])
def test_a_hypersonic_free_stream_against_the_oracle(tpp, precision):
    import oracle as O
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20", lambda: cg.naca0012_jittered(48, 20))
    s = lk.Solver(cloud, 6.0, 0.0, cfl=0.1, inner_iters=0, first_order_iters=1, precision=precision)
    s.set_launch_shape(tpp, 32)
    s.set_state(*_hypersonic(cloud.n, 4))
    U = s.field(lk.FIELD_U)
    s.run(1, check=False)
    ref, response = _density_response(O.Oracle(cloud), U, np.random.default_rng(5))
    # the first q-variable, up to 31 here, carries 1.5 units in its last place
    # (2^-48) on either side; two roundings each of the fluxes and weights
    rms = np.sqrt(np.mean((s.field(lk.FIELD_R) - ref) ** 2, axis=0))
    assert np.all(rms <= (2 * 1.5 * 2.0 ** -48 + 4 * 2.0 ** -53) * response), (rms, response)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tpp", [1, 4])
def test_a_batch_of_cases_in_and_out_of_the_ranges(tpp, precision):
    """Each case as alone, bit for bit: the hypersonic one by the FP64 kernel, the other by the fixed-point one."""
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20k", lambda: cg.naca0012_jittered(48, 20, kinetic_outer=True))
    conds = [(0.7, 1.0), (4.0, 0.0), (2.0, -1.0)]
    kw = dict(cfl=0.1, inner_iters=2, first_order_iters=100, precision=precision, farfield=lk.FARFIELD_KINETIC)
    b = lk.Solver.batch([cloud] * 3, conds, **kw)
    b.set_launch_shape(tpp, 32)
    b.run(4)
    U, R = (b.field(f).reshape(3, cloud.n, 4) for f in (lk.FIELD_U, lk.FIELD_R))
    launches = []
    for c, (m, a) in enumerate(conds):
        s = lk.Solver(cloud, m, a, **kw)
        s.set_launch_shape(tpp, 32)
        s.run(4)
        launches.append(s.info()["launches_per_iter"])
        assert np.array_equal(s.field(lk.FIELD_R), R[c]), c
        assert np.array_equal(s.field(lk.FIELD_U), U[c]), c
    # one residual kernel alone, both in the batch (and its repair kernel)
    assert launches[0] == launches[1] == launches[2] == b.info()["launches_per_iter"] - 2
