"""GPU: the default launch shape of single FP16 frames against the largest ring of 2 CTAs per SM, on both sides of the
list lengths where the default changes.  At 12 fragments per tile a ring of 70 KB, which then holds one item, took 1.27
times as long, at 16 1.14 times."""

import pytest

from frame_time import Frame
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 8, 9, 12, 16])
def test_default_shape_keeps_up_with_the_largest_ring(n):
    f = Frame(n, D.DFB_F16, tiles=32)
    default = f.shortest(lambda j, r: j + 0.5 * r)
    D.dfb_set_tuning(f.h, 110, 2, 1)
    largest = f.shortest(lambda j, r: j + 0.5 * r)
    f.close()
    assert default <= 1.1 * largest
