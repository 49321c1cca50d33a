"""GPU: BLEND_DEPTH with fragments that are empty at a pixel (depth +inf or NaN) but carry colour there, as renderers
without a depth buffer submit them: they are blended last, in list order.  Some of that colour is not finite, which
must reach the pixel as it does in a plain sort.  Lengths around the in-order loop's remainders and the staged fill.

Tolerance: each of the n blends rounds a value of at most 1 three times, at most 1.5 n units of 2^-24 (n = 17: 1.6e-6).
"""

import numpy as np
import pytest

from frame_time import Frame
from gpu_helpers import composite_once
from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 15, 16, 17])
@pytest.mark.parametrize("T", [8, 32])
@pytest.mark.parametrize("share", [0.5, 1.0])
def test_empty_fragments_with_colour(n, T, share):
    rng = np.random.default_rng([n, T])
    sc = scenes.random_scene(2 * T, 2 * T, T, [n] * 4, seed=n, alpha_max=0.3)
    z = np.empty_like(sc.depth)
    for t in range(4):
        at = np.nonzero(sc.tile_ids == t)[0]
        at = at[np.lexsort((at, sc.keys[at]))]
        z[at] = np.arange(len(at), dtype=np.float32)[:, None] + 1.0     # in list order
    empty = rng.random(z.shape) < share
    z[empty] = np.where(rng.random(empty.sum()) < 0.3, np.nan, np.inf)
    sc.depth[:] = z
    for dtype in (D.DFB_F32, D.DFB_F16, D.DFB_BF16, D.DFB_FP8E4M3):
        rgba = sc.rgba.copy()
        if dtype != D.DFB_FP8E4M3:                    # e4m3 has no infinity, and its scale would be one
            odd = empty & (rng.random(z.shape) < 0.02)
            rgba[odd, rng.integers(0, 4, odd.sum())] = rng.choice([np.inf, -np.inf, np.nan], odd.sum())
        stored, scales = scenes.store_rgba(rgba, dtype)
        fb = composite_once(sc, D.DFB_BLEND_DEPTH, stored, dtype, scales)
        with np.errstate(invalid="ignore"):
            want = o.composite_frame(sc.W, sc.H, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys,
                                     o.dequantize(stored, dtype, scales), sc.depth)
        got = fb.color()
        np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
        inf = np.isinf(want)
        np.testing.assert_array_equal(got[inf], want[inf])
        ok = np.isfinite(want)
        assert np.max(np.abs(got[ok] - want[ok]), initial=0.0) <= 1.5 * 17 * 2.0 ** -24
        fb.close()


def test_their_cost():
    """Blending them is a second look at the list and no sort: 0.55 times the composite of a frame in random order (as
    long as it, with a sort of every pixel that counts for each fragment)."""
    f = Frame(16, D.DFB_F16)
    empty = f.shortest(lambda j, r: j + float("inf"))
    random = f.shortest(lambda j, r: r)
    f.close()
    assert empty <= 0.8 * random
