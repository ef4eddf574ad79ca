"""The neighbour slots packed in threads: clouds on either side of every number
of threads have the same number of colours and levels whether their slots are
packed by one thread or several, and pass the layout's own check (no GPU)."""
import pytest

from paper_2406_07441_gb300 import cloudgen as cg
from paper_2406_07441_gb300 import lskum as lk


@pytest.mark.parametrize("ni,nj", [(40, 16), (62, 33), (64, 32), (66, 32), (96, 32), (128, 64), (130, 64)])
def test_small_clouds_validate(ni, nj):
    cloud = cg.naca0012_block(ni, nj)
    one = lk.validate([cloud], [(0.6, 1.0)])
    assert lk.validate([cloud] * 3, [(0.6, 1.0)] * 3) == one
