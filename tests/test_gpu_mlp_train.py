"""Loss and gradients of batches at the edges of the training kernel's tiles
(128 points) and of its grid (one tile, and more than one, per SM) against the
FP64 oracle with BF16 rounding at the kernel's rounding points.  Bars as in
test_gpu_mlp.py (normwise per layer, 2e-3); with few points one activation
that rounds the other way (2^-8 relative) is not averaged away: 1e-2 there."""
import numpy as np
import pytest

from oracle import mlp as OM
from tests.test_gpu_mlp import _random_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000, 152 * 128, 152 * 128 + 1, 40000])
def test_loss_and_gradients_at_the_edges(n):
    from paper_2406_07441_gb300 import lskum as lk
    rng = np.random.default_rng(n)
    m = lk.Mlp(seed=3, max_batch=n)
    p = _random_params(rng, 1.5)
    m.set_params(p)
    X = rng.normal(0, 1, (n, 34)).astype(np.float32)
    T = rng.normal(0, 0.3, (n, 4)).astype(np.float32)
    ref = OM.loss_and_grads(lk.unflatten_params(p.astype(np.float64)), X.astype(np.float64), T.astype(np.float64),
                            bf16_round=True)
    bar = 2e-3 if n >= 1000 else 1e-2
    loss, g = m.loss_grads(X, T)
    assert abs(loss - ref[0]) <= bar * ref[0]
    for (gW, gb), (rW, rb) in zip(lk.unflatten_params(g.astype(np.float64)), ref[1]):
        assert np.linalg.norm(gW - rW) <= bar * np.linalg.norm(rW)
        assert np.linalg.norm(gb - rb) <= bar * np.linalg.norm(rb)
    loss2, g2 = m.loss_grads(X, T)
    assert loss2 == loss and np.array_equal(g2, g)  # fixed order of all sums
