"""GPU: staged BLEND_DEPTH lists that are nearly in order (a pair of fragments swapped), wholly out of it, and with
empty fragments between: the sort takes two fragments at a time and counts only where one is nearer than one before it.
Lengths around the pairs' and the counting loop's remainders, up to the staged fill.

Tolerance: each of the n blends rounds a value of at most 1 three times, at most 1.5 n units of 2^-24 (n = 16: 1.5e-6).
"""

import numpy as np
import pytest

from frame_time import Frame
from gpu_helpers import composite_once
from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 5, 6, 9, 15, 16])
@pytest.mark.parametrize("order", ["first", "middle", "last", "reversed", "ends", "levels"])
def test_swapped_pairs(n, order):
    rng = np.random.default_rng([n, len(order)])
    T = 16
    sc = scenes.random_scene(2 * T, T, T, [n, n], seed=n, alpha_max=0.3)
    for t in range(2):
        at = np.nonzero(sc.tile_ids == t)[0]
        at = at[np.lexsort((at, sc.keys[at]))]
        z = np.repeat(np.arange(n, dtype=np.float32)[:, None] - 2.0, T * T, axis=1)
        i, j = {"first": (0, 1), "middle": ((n - 1) // 2, (n - 1) // 2 + 1), "last": (n - 2, n - 1),
                "ends": (0, n - 1)}.get(order, (0, 0))
        z[[i, j]] = z[[j, i]]
        if order == "reversed":
            z = z[::-1].copy()
        elif order == "levels":
            z = rng.integers(-1, 2, z.shape).astype(np.float32) * np.float32(0.5)
            z[z == 0] = np.where(rng.random((z == 0).sum()) < 0.5, -0.0, 0.0)
        if t:                                         # empty fragments anywhere, -inf too
            u = rng.random(z.shape)
            z[u < 0.1], z[(u >= 0.1) & (u < 0.2)], z[u > 0.97] = np.inf, np.nan, -np.inf
        sc.depth[at] = z
    for dtype in (D.DFB_F32, D.DFB_F16):
        stored, scales = scenes.store_rgba(sc.rgba, dtype)
        fb = composite_once(sc, D.DFB_BLEND_DEPTH, stored, dtype, scales)
        want = o.composite_frame(sc.W, sc.H, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys,
                                 o.dequantize(stored, dtype, scales), sc.depth)
        assert np.max(np.abs(fb.color() - want)) <= 1.5 * 16 * 2.0 ** -24
        fb.close()


def test_cost_of_nearly_sorted_lists():
    """16 fragments of which the last two are swapped take 1.5 times the composite of the frame in order (1.9 times,
    with a count for every fragment by itself)."""
    f = Frame(16, D.DFB_F32)
    near = f.shortest(lambda j, r: j + 2.0 * (j == 14) - 1.0 * (j >= 14))
    ordered = f.shortest(lambda j, r: j + 0.5 * r)
    f.close()
    assert near <= 1.7 * ordered
