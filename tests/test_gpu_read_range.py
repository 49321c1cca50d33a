"""GPU: reads into a device buffer that is too small for the image return DFB_ERR_CUDA and write nothing; one of
exactly the image's size is filled."""

import ctypes as C

import numpy as np
import pytest

from gpu_helpers import GpuFrameBuffer
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu
W, H, T = 160, 96, 4                                  # colour 240 KB, RGBA8 60 KB, 960 tiles: 3.75 KB of variances
FILL = 0xA5


@pytest.fixture
def slots():
    """Device allocations of 256 KB and those that another one of them follows, so that nothing but this test's own
    memory lies past the end."""
    import torch
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    cuda = C.CDLL("libcuda.so.1")
    size, got = 256 << 10, []
    for _ in range(12):
        p = C.c_uint64()
        assert cuda.cuMemAlloc_v2(C.byref(p), C.c_size_t(size)) == 0
        assert cuda.cuMemsetD8_v2(C.c_uint64(p.value), C.c_ubyte(FILL), C.c_size_t(size)) == 0
        got.append(p.value)
    torch.cuda.synchronize()

    def host(p):
        a = np.empty(size, np.uint8)
        assert cuda.cuMemcpyDtoH_v2(a.ctypes.data_as(C.c_void_p), C.c_uint64(p), C.c_size_t(size)) == 0
        return a

    pairs = [p for p in got if p + size in got]
    yield pairs, size, host
    for p in got:
        cuda.cuMemFree_v2(C.c_uint64(p))


@pytest.mark.parametrize("image", ["color", "rgba8", "tile_variance"])
@pytest.mark.parametrize("short", [0, 16, 4096])
def test_destination_too_small(slots, image, short):
    import torch
    pairs, size, host = slots
    if not pairs:
        pytest.skip("no two allocations follow one another")
    fb = GpuFrameBuffer(W, H, T, D.DFB_BLEND_DEPTH, bg=(0.25, 0.5, 0.75, 1.0))
    fb.begin(0)
    fb.end()
    D.dfb_sync(fb.h)
    read, want = {"color": (D.dfb_read_color, fb.color()), "rgba8": (D.dfb_read_rgba8, fb.rgba8()),
                  "tile_variance": (lambda h, o: D.dfb_read_variance(h, None, o), fb.variance()[1])}[image]
    want = want.view(np.uint8).reshape(-1)
    if short > len(want):
        pytest.skip("the image is smaller than that")
    at = pairs[0] + size - len(want) + short          # `short` bytes of the image lie past the allocation
    if short:
        with pytest.raises(D.DfbError) as e:
            read(fb.h, at)
        assert e.value.code == D.DFB_ERR_CUDA
        torch.cuda.synchronize()
        assert (host(pairs[0]) == FILL).all()
    else:
        read(fb.h, at)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(host(pairs[0])[size - len(want):], want)
    assert (host(pairs[0] + size) == FILL).all()
    fb.begin(0)                                       # the handle still works
    fb.end()
    np.testing.assert_array_equal(fb.color()[0, 0], np.float32([0.25, 0.5, 0.75, 1.0]))
    fb.close()
