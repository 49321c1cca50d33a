"""GPU: frames around the size up to which a frame's records travel as a kernel parameter (128 records, 128 tiles,
2^20 pixels of them), mixed with larger ones on one handle and on alternating streams, against the same frames ended
in a batch: the same bits in every buffer."""

import numpy as np
import pytest

from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu

# (W, H, T): 128 tiles, 129 tiles, 1 tile, 16 tiles of which 112 or more fragments pass 2^20 pixels
SIZES = [(128, 64, 8), (129 * 8, 8, 8), (64, 64, 64), (1024, 1024, 256), (250, 250, 64)]


@pytest.mark.parametrize("W,H,T", SIZES)
def test_small_and_large_frames_mixed(W, H, T):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(W + T)
    rng = np.random.default_rng(W + T)
    tiles = -(-W // T) * -(-H // T)
    one, both, other = (D.dfb_create_ex(w, h, T, D.DFB_BLEND_DEPTH, D.DFB_F32)
                        for w, h in ((W, H), (W, H), (T, T)))
    pool = torch.rand((130, T * T, 4), generator=gen, device="cuda") * 0.3
    depth = torch.rand((130, T * T), generator=gen, device="cuda")
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    D.dfb_set_timing(one, True)
    for f, n in enumerate([0, 1, 127, 128, 129, 128, 129, 130, 5, 40, 129, 3, 3, 3]):
        ids = rng.integers(0, tiles, n).astype(np.int32)
        if n > 100:
            ids[:20] = ids[0]                 # one long list: the exact re-do runs as well
        at = rng.permutation(130)[:n].astype(np.uint64)
        keys = rng.integers(0, 4, n).astype(np.float32)
        for h in (one, both, other):
            D.dfb_begin_frame(h, f % 5 != 0)
        for h in (one, both):
            D.dfb_submit_tiles(h, ids, keys, np.uint64(pool.data_ptr()) + at * np.uint64(T * T * 16),
                               np.uint64(depth.data_ptr()) + at * np.uint64(T * T * 4), None, D.DFB_PTR_DEVICE)
        D.dfb_end_frame(one, streams[f // 2 % 2])
        D.dfb_end_frames([both, other], streams[f // 3 % 2])
        if f % 3 != 1:                        # else the next frame follows without a read
            got = []
            for h in (one, both):
                a = [np.empty((H, W, 4), np.float32) for _ in range(3)] + [np.empty((H, W), np.uint32),
                                                                           np.empty(tiles, np.float32)]
                D.dfb_read_color(h, a[0])
                D.dfb_read_accum(h, a[1])
                D.dfb_read_variance(h, a[2], a[4])
                D.dfb_read_rgba8(h, a[3])
                got.append(a)
            for x, y in zip(*got):
                np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
    assert D.dfb_read_timing(one)["launches"] == 14
    for h in (one, both, other):
        D.dfb_destroy(h)
