"""GPU: the images of mean, variance and saved state, which kernels write, into device buffers that are too small
(DFB_ERR_CUDA, nothing written) and into ones whose address is no multiple of 16 (the same bits)."""

import numpy as np
import pytest

from gpu_helpers import GpuFrameBuffer
from harness import scenes
from paper_2305_07083_gb300 import dfb as D
from test_gpu_read_range import FILL, slots  # noqa: F401

pytestmark = pytest.mark.gpu
W, H, T = 160, 96, 16                                 # an image is 240 KB


def accumulated():
    sc = scenes.random_scene(W, H, T, [2] * 60, seed=3, alpha_max=0.5)
    fb = GpuFrameBuffer(W, H, T, D.DFB_BLEND_DEPTH)
    for f in range(2):
        fb.begin(f)
        fb.submit_pool(sc.tile_ids, sc.keys, sc.rgba * (1.0 - 0.3 * f), sc.depth)
        fb.end()
    D.dfb_sync(fb.h)
    state = [np.empty((H, W, 4), np.float32) for _ in range(3)]
    assert D.dfb_save_accum(fb.h, *state) == 2
    return fb, {"mean": fb.accum(), "variance": fb.variance()[0], "sum": state[0], "m2": state[2]}


def read(fb, image, at, spare):
    if image == "mean":
        D.dfb_read_accum(fb.h, at)
    elif image == "variance":
        D.dfb_read_variance(fb.h, at, None)
    else:
        D.dfb_save_accum(fb.h, *([at, spare, spare] if image == "sum" else [spare, spare, at]))


@pytest.mark.parametrize("image", ["mean", "variance", "sum", "m2"])
@pytest.mark.parametrize("short", [0, 16, 4096, -4, -12])
def test_too_small_or_unaligned(slots, image, short):  # noqa: F811
    import torch
    pairs, size, host = slots
    if not pairs:
        pytest.skip("no two allocations follow one another")
    fb, images = accumulated()
    want = images[image].view(np.uint8).reshape(-1)
    spare = torch.empty((H, W, 4), device="cuda")
    at = pairs[0] + size - len(want) + short          # `short` bytes of the image lie past the allocation
    if short > 0:
        with pytest.raises(D.DfbError) as e:
            read(fb, image, at, spare)
        assert e.value.code == D.DFB_ERR_CUDA
        torch.cuda.synchronize()
        assert (host(pairs[0]) == FILL).all()
    else:
        read(fb, image, at, spare)
        torch.cuda.synchronize()
        got = host(pairs[0])
        np.testing.assert_array_equal(got[size - len(want) + short:size + short], want)
        assert (got[:size - len(want) + short] == FILL).all() and (got[size + short:] == FILL).all()
    assert (host(pairs[0] + size) == FILL).all()
    fb.begin(1)                                       # the handle still works
    fb.end()
    D.dfb_sync(fb.h)
    fb.close()
