"""Contexts of different sizes side by side, each in a thread of its own, on one
GPU: re-captured, timed by phase and run at the same time, they get what each
gets alone, bit for bit, and no call fails (their sweeps' launches have
different numbers of warps, and so different amounts of shared memory)."""
import threading

import numpy as np
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu

CLOUDS = {
    "block_40x16": lambda: cg.naca0012_block(40, 16),
    "block_80x32": lambda: cg.naca0012_block(80, 32),
    "jit_48x20": lambda: cg.naca0012_jittered(48, 20),
    "jit336x136": lambda: cg.naca0012_jittered(336, 136),
}


def _work(cloud, precision, jvp, rounds):
    """Re-captures and phase timings (two launches of the sweeps each) in turn with iterations, from one state."""
    from paper_2406_07441_gb300 import lskum as lk
    s = lk.Solver(cloud, 0.63, 2.0, cfl=10.0, inner_iters=1, first_order_iters=10 ** 6, precision=precision, jvp=jvp)
    U = s.field(lk.FIELD_U)
    for r in range(rounds):
        s.set_launch_shape(2, (32, 4)[r & 1])
        s.set_conserved(U)
        s.time_phases(40)
        s.set_conserved(U)
        s.run(3)
    out = s.field(lk.FIELD_U)
    s.close()
    return out


@pytest.mark.parametrize("precision,jvp", [(0, 0), (1, 0), (0, 1)])
def test_contexts_in_threads_equal_themselves_alone(precision, jvp):
    rounds = 10
    clouds = [cached_cloud(name, make) for name, make in CLOUDS.items()]
    alone = [_work(c, precision, jvp, rounds) for c in clouds]
    got, failed = [None] * len(clouds), []

    def run(i):
        try:
            got[i] = _work(clouds[i], precision, jvp, rounds)
        except Exception as e:  # (reported by the main thread)
            failed.append((i, e))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(clouds))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for a, g in zip(alone, got):
        assert np.array_equal(a, g)
