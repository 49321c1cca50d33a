"""GPU: handles of one launch, or of a graph, outlive the handle or graph whose error word the launch reported to."""

import numpy as np
import pytest

from gpu_helpers import GpuFrameBuffer
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu
BG = (0.5, 0.25, 0.125, 1.0)


def frames(n):
    out = [GpuFrameBuffer(64, 32, 16, D.DFB_BLEND_DEPTH, bg=BG) for _ in range(n)]
    for fb in out:
        fb.begin(0)
    return out


def check(fb):
    D.dfb_sync(fb.h)
    np.testing.assert_array_equal(fb.color().reshape(-1, 4), np.tile(np.float32(BG), (64 * 32, 1)))


@pytest.mark.parametrize("first", [0, 1, 2])
def test_batch(first):
    fbs = frames(3)
    D.dfb_end_frames([fb.h for fb in fbs])
    order = [first] + [i for i in range(3) if i != first]
    for k, i in enumerate(order):
        for j in order[k:]:
            check(fbs[j])
        fbs[i].close()


def test_graph():
    fbs = frames(2)
    g = D.dfb_graph_create([fb.h for fb in fbs])
    D.dfb_graph_launch(g)
    check(fbs[0])
    D.dfb_graph_destroy(g)
    for fb in fbs:
        check(fb)
        fb.begin(1)
        fb.end()
        check(fb)
        fb.close()
