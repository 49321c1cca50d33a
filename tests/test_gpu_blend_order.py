"""GPU: BLEND_DEPTH's in-order pass and its exact fall-backs, at list lengths around the unrolled loop's remainders,
the staged fill (16) and the fills of 8, in full (256-pixel) and small items.

Tolerance: each of the n blends rounds a value of at most 1 three times (weight, product and sum), so at most 1.5 n
units of 2^-24; the longest list here has 33 fragments: 3e-6.
"""

import numpy as np
import pytest

from gpu_helpers import composite_once
from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu
TOL = 1.5 * 33 * 2.0 ** -24


def scene(T, n, seed):
    """One frame of 4 tiles: depths in key order with, at some pixels, empty fragments (zero and not zero), equal
    depths, and a pair out of order."""
    sc = scenes.random_scene(2 * T, 2 * T, T, [n, max(n - 1, 0), 1, 0], seed=seed, alpha_max=0.3)
    rng = np.random.default_rng(seed)
    for t in range(4):
        at = np.nonzero(sc.tile_ids == t)[0]
        at = at[np.lexsort((at, sc.keys[at]))]
        if len(at) == 0:
            continue
        z = np.sort(rng.integers(0, 3 * len(at), (len(at), T * T)), axis=0).astype(np.float32)
        u = rng.random(z.shape)
        rgba = sc.rgba[at]
        empty = u < 0.2
        z[empty] = np.where(rng.random(empty.sum()) < 0.3, np.nan, np.inf)
        rgba[empty] = 0.0
        odd = (u < 0.001) & empty                        # empty, but not zero
        rgba[odd] = (0.2, 0.1, 0.05, 0.25)
        for p in np.nonzero(rng.random(T * T) < 0.02)[0]:
            i, j = rng.integers(0, len(at), 2)
            z[[i, j], p] = z[[j, i], p]
        sc.depth[at] = z
        sc.rgba[at] = rgba
    return sc


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 23, 24, 25, 33])
@pytest.mark.parametrize("T", [8, 32])
def test_depth_order(n, T):
    sc = scene(T, n, 100 * n + T)
    for dtype in (D.DFB_F32, D.DFB_F16, D.DFB_BF16, D.DFB_FP8E4M3):
        stored, scales = scenes.store_rgba(sc.rgba, dtype)
        fb = composite_once(sc, D.DFB_BLEND_DEPTH, stored, dtype, scales)
        want = o.composite_frame(sc.W, sc.H, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys,
                                 o.dequantize(stored, dtype, scales), sc.depth)
        assert np.max(np.abs(fb.color() - want)) <= TOL
        fb.close()
