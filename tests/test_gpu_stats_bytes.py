"""GPU: dfb_frame_stats.fragment_bytes against a count per tile: RGBA of every fragment, depth where a mode reads it.
BLEND_DEPTH does not read the depth of a tile's only fragment."""

import numpy as np
import pytest

from gpu_helpers import GpuFrameBuffer, to_dev
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,T", [(70, 40, 16), (64, 64, 64), (16, 16, 32), (96, 33, 32), (33, 96, 4)])
@pytest.mark.parametrize("dtype", [D.DFB_F32, D.DFB_F16, D.DFB_FP8E4M3])
@pytest.mark.parametrize("prepared", [False, True])
def test_fragment_bytes(W, H, T, dtype, prepared):
    rng = np.random.default_rng([W, H, T])
    tx, ty = -(-W // T), -(-H // T)
    counts = rng.choice([0, 1, 1, 2, 17], tx * ty)
    ids = np.repeat(np.arange(tx * ty, dtype=np.int32), counts)
    ids = ids[rng.permutation(len(ids))]
    n, eb = len(ids), D.ELEMENT_BYTES[dtype]
    pixels = np.array([min(T, W - t % tx * T) * min(T, H - t // tx * T) for t in range(tx * ty)], np.int64)
    rgba = to_dev(np.zeros((max(n, 1), T * T * 4 * eb), np.uint8))
    depth = to_dev(np.zeros((max(n, 1), T * T), np.float32))
    args = (ids, np.zeros(n, np.float32), D.pool_pointers(rgba, n, T * T * 4 * eb),
            D.pool_pointers(depth, n, T * T * 4), np.ones(n, np.float32) if dtype == D.DFB_FP8E4M3 else None)
    for mode, read in ((D.DFB_BLEND_DEPTH, counts * (counts > 1)), (D.DFB_BLEND_ORDERED, 0 * counts)):
        fb = GpuFrameBuffer(W, H, T, mode, dtype)
        if prepared and n:
            s = D.dfb_tileset_create(fb.h, *args)
            D.dfb_run_frames([fb.h], [s], [0])
            D.dfb_sync(fb.h)
            D.dfb_tileset_destroy(s)
        else:
            fb.begin(0)
            if n:
                D.dfb_submit_tiles(fb.h, *args, D.DFB_PTR_DEVICE)
            fb.end()
        assert fb.stats()["fragment_bytes"] == int((pixels * (counts * 4 * eb + read * 4)).sum())
        fb.close()
