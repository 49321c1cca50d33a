"""GPU: reads into device memory captured in a graph: the images of a frame with contents, into destinations that
hold other values before each replay."""

import numpy as np
import pytest

from gpu_helpers import GpuFrameBuffer
from harness import scenes
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["relaxed", "global"])
def test_captured_reads_fill_their_destinations(mode):
    import torch
    W, H, T = 257, 255, 32
    sc = scenes.random_scene(W, H, T, [3] * 72, seed=5, alpha_max=0.5)
    fb = GpuFrameBuffer(W, H, T, D.DFB_BLEND_DEPTH, bg=(0.1, 0.2, 0.3, 0.5))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for f in range(2):
        fb.begin(f)
        fb.submit_pool(sc.tile_ids, sc.keys, sc.rgba * (1.0 - 0.3 * f), sc.depth)
        fb.end(s)
    want = [fb.color(), fb.accum(), fb.rgba8(), fb.variance()[0], fb.variance()[1]]
    for w in want:
        assert np.count_nonzero(w.view(np.int32)) > w.size // 2
    D.dfb_sync(fb.h)
    out = [torch.empty(w.shape, dtype=torch.int32, device="cuda") for w in want]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode=mode):
        D.dfb_read_color(fb.h, out[0])
        D.dfb_read_accum(fb.h, out[1])
        D.dfb_read_rgba8(fb.h, out[2])
        D.dfb_read_variance(fb.h, out[3], out[4])
    for _ in range(2):
        for o in out:
            o.fill_(-7)
        g.replay()
        torch.cuda.synchronize()
        for o, w in zip(out, want):
            np.testing.assert_array_equal(o.cpu().numpy(), w.view(np.int32))
    fb.close()
