"""Device memory of a context: the per-point lower and upper lists are kept
only where a kernel reads them (lists too long for the packed sweeps)."""
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from tests.conftest import cached_cloud

pytestmark = pytest.mark.gpu


def test_packed_contexts_hold_no_lists_by_point():
    torch = pytest.importorskip("torch")
    from paper_2406_07441_gb300 import lskum as lk
    cloud = cached_cloud("naca640x256_jit", lambda: cg.naca0012_jittered(640, 256))
    n, nnz = cloud.n, cloud.nnz
    lk.Solver(cloud, 0.8, 1.0).close()  # (the library's own memory)
    free = torch.cuda.mem_get_info()[0]
    s = lk.Solver(cloud, 0.8, 1.0)
    used = free - torch.cuda.mem_get_info()[0]
    s.close()
    # per slot: index 4, membership 1, half offsets 16, weights 16 (residual),
    # 16 and 32 (q-derivatives), the packed lists' index and membership 4 and
    # weights 16, with a tenth for padding (framed points: indexes, weights and
    # a Jacobian, 16 doubles, of which there are 2 % of the points); per point:
    # two states of (4 + 4 + 24 doubles, 4 integers), three derivatives (8
    # doubles and 4 int4), geometry 20 doubles, increments, R, D, products and
    # the scratch 42 doubles, the rest below 200 bytes.  The lists by point
    # would add 21 bytes per slot.
    slot = 1.1 * (4 + 1 + 16 + 16 + 16 + 32 + 4 + 16)
    framed = 0.02 * n * (nnz / n) * 2 * (37 + 128) + 0.02 * n * 512
    point = 2 * (36 * 8) + 3 * (64 + 64) + 20 * 8 + 42 * 8 + 200
    assert used < nnz * slot + n * point + framed + (16 << 20), (used, nnz * slot, n * point, framed)
