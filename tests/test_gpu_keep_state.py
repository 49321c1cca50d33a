"""GPU: an accumulating frame larger than L2, ended alone (its state partly kept in L2, everything else streamed) and
ended together with another frame (ordinary accesses): the same bits in every buffer, with the state streamed through
the ring (1 fragment per tile) and loaded by the consumers (3 per tile), Kahan-compensated from the second frame on."""

import numpy as np
import pytest

from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu
W, H, T = 1600, 1080, 64          # at least 116 MB per frame; ragged in both directions


@pytest.mark.parametrize("per_tile", [1, 3])
@pytest.mark.parametrize("dtype", [D.DFB_F32, D.DFB_FP8E4M3])
def test_alone_equals_together(dtype, per_tile):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7 * per_tile + dtype)
    tiles = -(-W // T) * -(-H // T)
    n = tiles * per_tile
    ids = np.tile(np.arange(tiles, dtype=np.int32), per_tile)
    keys = np.repeat(np.arange(per_tile, dtype=np.float32), tiles)
    depth = torch.rand((n, T * T), generator=gen, device="cuda").contiguous()
    scales = np.full(n, 1.0 / 448.0, np.float32) if dtype == D.DFB_FP8E4M3 else None
    one, both, other = (D.dfb_create_ex(w, h, T, D.DFB_BLEND_DEPTH, dtype, D.DFB_FLAGS_DEFAULT, 1)
                        for w, h in ((W, H), (W, H), (T, T)))
    keep = []
    for f in range(4):
        rgba = torch.rand((n, T * T, 4), generator=gen, device="cuda") * 0.4
        if dtype == D.DFB_FP8E4M3:
            rgba = (rgba * 448.0).to(torch.float8_e4m3fn)
        keep.append(rgba)
        for h in (one, both, other):
            D.dfb_begin_frame(h, f > 0)
        for h in (one, both):
            D.dfb_submit_tiles(h, ids, keys, D.pool_pointers(rgba, n, T * T * 4 * D.ELEMENT_BYTES[dtype]),
                               D.pool_pointers(depth, n, T * T * 4), scales, D.DFB_PTR_DEVICE)
        D.dfb_end_frame(one, None)
        D.dfb_end_frames([both, other], None)
    got = []
    for h in (one, both):
        a = [np.empty((H, W, 4), np.float32) for _ in range(4)]
        px8, per = np.empty((H, W), np.uint32), np.empty(tiles, np.float32)
        assert D.dfb_save_accum(h, a[0], a[1], a[2]) == 4
        D.dfb_read_color(h, a[3])
        D.dfb_read_rgba8(h, px8)
        D.dfb_read_variance(h, None, per)
        got.append(a + [px8, per])
    for x, y in zip(*got):
        np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
    assert np.abs(got[0][1]).max() > 0       # the compensation ran
    for h in (one, both, other):
        D.dfb_destroy(h)
