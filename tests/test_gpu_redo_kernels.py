"""GPU: the two kernels of the exact re-do, each over its own units: launches that have lists for one of them, for both
and in several frames at once, against the oracle, and the number of kernels that a frame reports.

Tolerance: each of the n blends rounds a value of at most 1 three times, at most 1.5 n units of 2^-24 (n = 70: 6.3e-6).
"""

import numpy as np
import pytest

from frame_time import Frame
from gpu_helpers import GpuFrameBuffer, to_dev
from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu
TOL = 1.5 * 70 * 2.0 ** -24


@pytest.mark.parametrize("counts,kernels", [([17, 3], 1), ([48, 16], 1), ([49, 16], 1), ([48, 49], 2), ([70, 17], 2),
                                            ([16, 16], 0)])
@pytest.mark.parametrize("T", [8, 32])
def test_one_kernel_or_both(counts, kernels, T):
    sc = scenes.random_scene(2 * T, T, T, counts, seed=sum(counts), alpha_max=0.2, special_depths=True)
    want = o.composite_frame(sc.W, sc.H, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys, sc.rgba, sc.depth)
    fb = GpuFrameBuffer(sc.W, sc.H, T, D.DFB_BLEND_DEPTH)
    for f in range(3):
        before = fb.stats()["kernel_launches"] if f else 0
        fb.begin(f)
        fb.submit_pool(sc.tile_ids, sc.keys, sc.rgba, sc.depth)
        fb.end()
        assert np.max(np.abs(fb.color() - want)) <= TOL
        assert fb.stats()["kernel_launches"] - before == 3 + kernels
    assert np.max(np.abs(fb.accum() - want)) <= 2 * TOL
    fb.close()


def test_frames_in_one_launch():
    T, frames = 16, []
    for counts in ([60, 5], [20, 48], [3, 1], [49, 17]):
        sc = scenes.random_scene(2 * T, T, T, counts, seed=sum(counts), alpha_max=0.2)
        fb = GpuFrameBuffer(sc.W, sc.H, T, D.DFB_BLEND_DEPTH)
        fb.begin(0)
        fb.submit_pool(sc.tile_ids, sc.keys, sc.rgba, sc.depth)
        frames.append((sc, fb))
    D.dfb_end_frames([fb.h for _, fb in frames])
    for sc, fb in frames:
        want = o.composite_frame(sc.W, sc.H, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys, sc.rgba, sc.depth)
        assert np.max(np.abs(fb.color() - want)) <= TOL
    for _, fb in reversed(frames):
        fb.close()


@pytest.mark.parametrize("counts", [[60, 5], [20, 48], [49, 17]])
def test_allocation_free_call(counts):
    import torch
    T = 16
    sc = scenes.random_scene(2 * T, T, T, counts, seed=sum(counts), alpha_max=0.2)
    rgba, depth, n = to_dev(sc.rgba), to_dev(sc.depth), len(sc.tile_ids)
    out = torch.empty((T, 2 * T, 4), device="cuda")
    torch.cuda.synchronize()
    D.dfb_composite_noalloc(2 * T, T, T, D.DFB_BLEND_DEPTH, D.DFB_F32, sc.tile_ids, sc.keys,
                            D.pool_pointers(rgba, n, T * T * 16), D.pool_pointers(depth, n, T * T * 4), None, None, out,
                            None, torch.cuda.current_stream())
    want = o.composite_frame(2 * T, T, T, o.BLEND_DEPTH, sc.tile_ids, sc.keys, sc.rgba, sc.depth)
    assert np.max(np.abs(out.cpu().numpy() - want)) <= TOL


def test_cost_of_the_longer_lists():
    """A frame out of order everywhere takes 1.45 times as long with 49 fragments per tile, in windowed rounds, as with
    48, ranked (1.9 times with both in one kernel)."""
    times = []
    for n in (48, 49):
        f = Frame(n, D.DFB_F32, tiles=8)
        times.append(f.shortest(lambda j, r: r, frames=20, whole=True))
        f.close()
    assert times[1] <= 1.7 * times[0]
