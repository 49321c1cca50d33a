"""GPU: reads of a frame's buffers into device memory against the same reads into host memory (a copy of the same
bits): odd pixel counts (the copy kernel's remainder), destinations that are not 16-byte aligned (plain copy),
nothing written outside, and reads captured in a graph."""

import numpy as np
import pytest

from harness import scenes
from gpu_helpers import GpuFrameBuffer
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


def frame(W, H, T):
    sc = scenes.random_scene(W, H, T, [3] * (-(-W // T) * -(-H // T)), seed=W * H, alpha_max=0.5)
    fb = GpuFrameBuffer(W, H, T, D.DFB_BLEND_DEPTH)
    for f in range(2):
        fb.begin(f)
        fb.submit_pool(sc.tile_ids, sc.keys, sc.rgba * (1.0 - 0.3 * f), sc.depth)
        fb.end()
    return fb


@pytest.mark.parametrize("W,H,T", [(1, 1, 4), (37, 29, 16), (64, 64, 64), (257, 255, 32), (1031, 517, 64)])
@pytest.mark.parametrize("offset", [0, 1, 4])
def test_device_equals_host(W, H, T, offset):
    import torch
    fb = frame(W, H, T)
    color, px8 = fb.color(), fb.rgba8()
    mean = fb.accum()
    var, per = fb.variance()
    for want, read in ((color, D.dfb_read_color), (px8, D.dfb_read_rgba8), (mean, D.dfb_read_accum),
                       (per, lambda h, o: D.dfb_read_variance(h, None, o)),
                       (var, lambda h, o: D.dfb_read_variance(h, o, None))):
        if offset % 4 and (want is mean or want is var):
            continue                                  # written as float4: 16-byte aligned destinations only
        buf = torch.full((want.size + offset + 8,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        read(fb.h, buf.data_ptr() + 4 * offset)
        torch.cuda.synchronize()
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[offset:offset + want.size], want.view(np.int32).reshape(-1))
        assert (got[:offset] == -1).all() and (got[offset + want.size:] == -1).all()
    fb.close()


def test_reads_captured_in_a_graph():
    import torch
    fb = frame(257, 255, 32)
    s = torch.cuda.Stream()
    fb.begin(0)
    fb.end(s)                                         # the handle's last stream
    torch.cuda.synchronize()
    out = [torch.zeros((255, 257, 4), device="cuda") for _ in range(2)]
    px8 = torch.zeros((255, 257), dtype=torch.int32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        D.dfb_read_color(fb.h, out[0])
        D.dfb_read_accum(fb.h, out[1])
        D.dfb_read_rgba8(fb.h, px8)
    empty = fb.color(), fb.accum(), fb.rgba8()        # an empty frame
    g.replay()
    torch.cuda.synchronize()
    for got, w in zip(out + [px8], empty):
        np.testing.assert_array_equal(got.cpu().numpy().view(np.int32), w.view(np.int32))
    fb.close()
