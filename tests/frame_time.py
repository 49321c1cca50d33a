"""The time of a frame's composite, for tests that compare two kinds of frame with each other."""

from __future__ import annotations

import numpy as np

from paper_2305_07083_gb300 import dfb as D


class Frame:
    """`tiles` x `tiles` image tiles of 64x64 with n FP32 or FP16 fragments each, keys ascending; `order(j, r)` gives
    the depths from the place j in the list and a random number r per pixel."""

    def __init__(self, n, dtype, tiles=16):
        import torch
        self.n, self.count, self.dtype = n, tiles * tiles * n, dtype
        self.ids = np.repeat(np.arange(tiles * tiles, dtype=np.int32), n)
        self.keys = np.tile(np.arange(n, dtype=np.float32), tiles * tiles)
        kind = {D.DFB_F32: torch.float32, D.DFB_F16: torch.float16}[dtype]
        self.rgba = (torch.rand((self.count, 4096, 4), device="cuda") * 0.1).to(kind)
        self.j = torch.as_tensor(self.keys, device="cuda")[:, None]
        self.r = torch.rand((self.count, 4096), device="cuda")
        self.h = D.dfb_create_ex(64 * tiles, 64 * tiles, 64, D.DFB_BLEND_DEPTH, dtype, D.DFB_FLAG_WRITE_COLOR)
        D.dfb_set_timing(self.h, True)

    def close(self):
        D.dfb_destroy(self.h)

    def shortest(self, order, frames=40, whole=False):
        """Shortest composite of `frames` frames in ms, from the library's events around the launch; `whole`: all of a
        frame's kernels, from events around its end."""
        import torch
        depth = order(self.j, self.r).expand(self.count, 4096).contiguous()
        rgba = D.pool_pointers(self.rgba, self.count, 4096 * 4 * D.ELEMENT_BYTES[self.dtype])
        z = D.pool_pointers(depth, self.count, 4096 * 4)
        torch.cuda.synchronize()
        best, s = np.inf, torch.cuda.Stream()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for _ in range(frames):
            D.dfb_begin_frame(self.h, 0)
            D.dfb_submit_tiles(self.h, self.ids, self.keys, rgba, z, None, D.DFB_PTR_DEVICE)
            a.record(s)
            D.dfb_end_frame(self.h, s)
            b.record(s)
            b.synchronize()
            composite = D.dfb_read_timing(self.h)["composite_ms"]
            best = min(best, a.elapsed_time(b) if whole else composite)
        return best
