"""GPU: the exact re-do of long lists whose depths are out of list order, at list lengths around its batches (4 and
8), the longest list it ranks (48) and the window of the longer ones (16), against the oracle.

Tolerance: each of the n blends rounds a value of at most 1 three times, at most 1.5 n units of 2^-24 (n = 80: 7.2e-6).
"""

import numpy as np
import pytest

from gpu_helpers import composite_once
from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [17, 24, 25, 31, 32, 33, 47, 48, 49, 64, 80])
@pytest.mark.parametrize("dtype", [D.DFB_F32, D.DFB_F16, D.DFB_FP8E4M3])
def test_long_lists_out_of_order(n, dtype):
    sc = scenes.random_scene(70, 40, 32, [n, 2, n, n - 1, 0, 17], seed=n, alpha_max=0.2, special_depths=True,
                             depth_levels=None if n % 2 else 9)
    stored, scales = scenes.store_rgba(sc.rgba, dtype)
    fb = composite_once(sc, D.DFB_BLEND_DEPTH, stored, dtype, scales)
    want = o.composite_frame(70, 40, 32, o.BLEND_DEPTH, sc.tile_ids, sc.keys, o.dequantize(stored, dtype, scales),
                             sc.depth)
    assert np.max(np.abs(fb.color() - want)) <= 1.5 * 80 * 2.0 ** -24
    fb.close()
