"""Sweeps of clouds with long lower or upper lists against the oracle: more
than 32 slots, which only the form with one launch per level takes (2, 4 and 8
lanes per point); and 21 to 32 in levels wide enough for two lanes per point,
where a lane's share of the list exceeds what it loads ahead.  The kinetic far
field's packed sweeps against the oracle in both of their shapes."""
import numpy as np
import pytest

import oracle as O
from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud
from tests.wide import longest_list, two_rings

pytestmark = pytest.mark.gpu


def nrel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


# FP64: the bar of the other parity tests.  FP32 sweeps: theirs of 1e-5 holds for
# sums of up to 20 neighbours; here up to 87.
BAR = {0: 1e-10, 1: 1e-5 * 87 / 20}


def _check(s, r, precision):
    from paper_2406_07441_gb300 import lskum as lk
    assert nrel(s.field(lk.FIELD_R), r["R"]) < 1e-10
    assert nrel(s.field(lk.FIELD_DUS), r["dUs"]) < BAR[precision]
    assert nrel(s.field(lk.FIELD_DU), r["dU"]) < BAR[precision]


@pytest.mark.parametrize("lanes", [2, 4, 8])
@pytest.mark.parametrize("jvp,precision,lusgs", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (1, 1, 0), (0, 0, 1), (1, 0, 1)])
def test_one_launch_per_level(jvp, precision, lusgs, lanes):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("wide_48x20", lambda: two_rings(cg.naca0012_jittered(48, 20)))
    o = O.Oracle(cloud)
    assert longest_list(cloud, o.order) > 32
    kw = dict(cfl=2.0, K=1, jvp=jvp, first_order=10)
    U0 = o.initial_state(0.63, 2.0)
    r = o.run_manish(U0, 3, sigma=-1, **kw) if lusgs else o.run(U0, 3, **kw)
    assert r["status"] == 0
    s = lk.Solver(cloud, 0.63, 2.0, cfl=2.0, inner_iters=1, first_order_iters=10, jvp=jvp, precision=precision,
                  lusgs=lusgs)
    with pytest.raises(lk.LskumError) as e:
        s.set_launch_shape(2, 32)  # (no packed form of such lists)
    assert e.value.status == lk.ERR_ARG
    s.set_launch_shape(2, lanes)
    assert s.run(3) == 3
    if precision == 0:
        _check(s, r, 0)
    else:  # (three FP32 iterations: each adds its own error to the state)
        assert nrel(s.field(lk.FIELD_DU), r["dU"]) < 3 * BAR[1]


@pytest.mark.parametrize("lanes", [2, 8])
def test_one_launch_per_level_kinetic_far_field(lanes):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("wide_48x20k", lambda: two_rings(cg.naca0012_jittered(48, 20, kinetic_outer=True)))
    o = O.Oracle(cloud, farfield=O.FARFIELD_KINETIC, mach=1.2, aoa_deg=0.0)
    r = o.run(o.initial_state(1.2, 0.0), 2, cfl=2.0, K=1, first_order=10)
    assert r["status"] == 0
    s = lk.Solver(cloud, 1.2, 0.0, cfl=2.0, inner_iters=1, first_order_iters=10, farfield=lk.FARFIELD_KINETIC)
    s.set_launch_shape(2, lanes)
    assert s.run(2) == 2
    _check(s, r, 0)


@pytest.mark.parametrize("jvp,precision", [(0, 0), (1, 0), (0, 1)])
def test_wide_levels_with_more_slots_than_are_loaded_ahead(jvp, precision):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("wide_block", lambda: two_rings(cg.naca0012_block(400, 160)))
    key = "wide_block_oracle"
    o = cached_cloud(key, lambda: O.Oracle(cloud))
    # a level (colour) of more than 152 x 4 x 8 interior points, of which some
    # have more than 2 x 10 slots on one side of the sweep order
    pos = np.empty(cloud.n, np.int64)
    pos[o.order] = np.arange(cloud.n)
    own = np.repeat(np.arange(cloud.n), np.diff(cloud.nbr_off))
    swept = np.asarray(cloud.flag)[cloud.nbr_idx] != cg.OUTER
    lower = np.bincount(own, (pos[cloud.nbr_idx] < pos[own]) & swept, cloud.n)
    upper = np.bincount(own, (pos[cloud.nbr_idx] > pos[own]) & swept, cloud.n)
    inner = np.asarray(cloud.flag) == 0
    sizes = np.bincount(o.colour[inner])
    long = inner & (np.maximum(lower, upper) > 20) & (sizes[np.minimum(o.colour, sizes.size - 1)] > 4864)
    assert long.sum() > 1000 and max(lower.max(), upper.max()) <= 32
    U0 = o.initial_state(0.63, 2.0)
    r = cached_cloud(f"{key}_{jvp}", lambda: o.run(U0, 1, cfl=100.0, K=1, jvp=jvp, first_order=10))
    s = lk.Solver(cloud, 0.63, 2.0, inner_iters=1, first_order_iters=10, jvp=jvp, precision=precision)
    for shape in ((1, 32), (4, 4)):
        s.set_launch_shape(*shape)
        s.set_conserved(U0)
        assert s.run(1) == 1
        _check(s, r, precision)


@pytest.mark.parametrize("lanes", [4, 32])
@pytest.mark.parametrize("jvp", [0, 1])
def test_packed_kinetic_sweeps_against_the_oracle(jvp, lanes):
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("jit_48x20k11", lambda: cg.naca0012_jittered(48, 20, seed=11, kinetic_outer=True))
    o = O.Oracle(cloud, farfield=O.FARFIELD_KINETIC, mach=1.2, aoa_deg=0.0)
    r = o.run(o.initial_state(1.2, 0.0), 3, cfl=100.0, K=2, jvp=jvp, first_order=10)
    assert r["status"] == 0
    s = lk.Solver(cloud, 1.2, 0.0, inner_iters=2, first_order_iters=10, jvp=jvp, farfield=lk.FARFIELD_KINETIC)
    s.set_launch_shape(2, lanes)
    assert s.run(3) == 3
    _check(s, r, 0)
