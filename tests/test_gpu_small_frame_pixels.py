"""GPU: frames of 256x256 tiles on both sides of the pixel limit up to which a frame's records travel as a kernel
parameter, (records + tiles) * T * T <= 2^20: with 4 tiles 12 records do and 13 do not.  Mixed on one handle and on
alternating streams, against the same frames ended in a batch: the same bits in every buffer."""

import numpy as np
import pytest

from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,limit", [(512, 512, 12), (500, 300, 12), (256, 200, 15)])
def test_pixel_limit(W, H, limit):
    import torch
    T = 256
    gen = torch.Generator(device="cuda")
    gen.manual_seed(W + H)
    rng = np.random.default_rng(W + H)
    tiles = -(-W // T) * -(-H // T)
    assert (limit + tiles) * T * T == 2 ** 20
    one, both, other = (D.dfb_create_ex(w, h, T, D.DFB_BLEND_DEPTH, D.DFB_F32) for w, h in ((W, H), (W, H), (T, T)))
    pool = torch.rand((limit + 2, T * T, 4), generator=gen, device="cuda") * 0.3
    depth = torch.rand((limit + 2, T * T), generator=gen, device="cuda")
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for f, n in enumerate([limit, limit + 1, limit, limit, limit + 1, limit + 1, 1, limit + 2, 0, limit]):
        ids = rng.integers(0, tiles, n).astype(np.int32)
        at = rng.permutation(limit + 2)[:n].astype(np.uint64)
        keys = rng.integers(0, 4, n).astype(np.float32)
        for h in (one, both, other):
            D.dfb_begin_frame(h, f % 4 != 0)
        for h in (one, both):
            D.dfb_submit_tiles(h, ids, keys, np.uint64(pool.data_ptr()) + at * np.uint64(T * T * 16),
                               np.uint64(depth.data_ptr()) + at * np.uint64(T * T * 4), None, D.DFB_PTR_DEVICE)
        D.dfb_end_frame(one, streams[f // 2 % 2])
        D.dfb_end_frames([both, other], streams[f // 3 % 2])
        if f % 3 == 1:                                # the next frame follows without a read
            continue
        got = []
        for h in (one, both):
            a = [np.empty((H, W, 4), np.float32) for _ in range(3)] + [np.empty(tiles, np.float32)]
            D.dfb_read_color(h, a[0])
            D.dfb_read_accum(h, a[1])
            D.dfb_read_variance(h, a[2], a[3])
            got.append(a)
        for x, y in zip(*got):
            np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
        assert n == 0 or np.count_nonzero(got[0][0])
    for h in (one, both, other):
        D.dfb_destroy(h)
