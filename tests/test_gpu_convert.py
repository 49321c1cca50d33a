"""GPU: dfb_convert_tiles over the tile sizes and alignments its kernels differ by, bit for bit.

The casts round to nearest even and the FP8 code is the rounding of one correctly rounded FP32 quotient, so the
expected values are exact: no tolerance.
"""

import numpy as np
import pytest

from harness import scenes
from oracle import dfb_oracle as o
from paper_2305_07083_gb300 import dfb as D

pytestmark = pytest.mark.gpu


def tiles(n, pixels, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((n, pixels, 4)) * rng.uniform(1e-3, 600.0, (n, 1, 1))).astype(np.float32)
    x[n // 2] = 0.0                               # an all-zero tile
    x[-1, -1, -1] = 1e4                           # the last value of the pool decides a scale
    x[0, 0, 0] = -3e4                             # and the first one
    return x


def convert(x, dtype, src_off=0, dst_off=0):
    """Values `src_off` floats into one buffer -> codes `dst_off` bytes into another, and the scales."""
    import torch
    n, pixels = x.shape[:2]
    src = torch.zeros(x.size + src_off, device="cuda")
    src[src_off:] = torch.from_numpy(x.reshape(-1)).cuda()
    size = x.size * D.ELEMENT_BYTES[dtype]
    dst = torch.full((dst_off + size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    sc = torch.zeros(n, device="cuda")
    D.dfb_convert_tiles(src.data_ptr() + 4 * src_off, dst.data_ptr() + dst_off, sc, n, pixels, dtype)
    torch.cuda.synchronize()
    got = dst.cpu().numpy()
    assert (got[:dst_off] == 0xA5).all() and (got[dst_off + size:] == 0xA5).all()   # nothing written outside
    return got[dst_off:dst_off + size], sc.cpu().numpy()


def check(x, dtype, **kw):
    got, scales = convert(x, dtype, **kw)
    if dtype == D.DFB_FP8E4M3:
        for t in range(len(x)):
            codes, s = o.fp8_quantize_tile(x[t])
            assert scales[t] == s
            np.testing.assert_array_equal(got.reshape(len(x), -1)[t], codes.reshape(-1))
    else:
        want, _ = scenes.store_rgba(x, dtype)
        np.testing.assert_array_equal(got.view(np.uint16), want.view(np.uint16).reshape(-1))


# 16 to 16384 pixels: tiles kept in registers by 2 threads up to a cluster of four CTAs; the tile counts leave the
# last CTA partly empty.  65536 and the others: the general kernel.
@pytest.mark.parametrize("n,pixels", [(257, 16), (65, 64), (17, 256), (5, 1024), (3, 4096), (2, 16384), (1, 16384),
                                      (2, 65536), (3, 1), (7, 5), (3, 1023)])
@pytest.mark.parametrize("dtype", [D.DFB_F16, D.DFB_BF16, D.DFB_FP8E4M3])
def test_tile_sizes(n, pixels, dtype):
    check(tiles(n, pixels, n * 7 + pixels), dtype)


@pytest.mark.parametrize("src_off,dst_off", [(1, 0), (0, 2), (2, 8)])
@pytest.mark.parametrize("dtype", [D.DFB_F16, D.DFB_BF16, D.DFB_FP8E4M3])
def test_unaligned(src_off, dst_off, dtype):
    check(tiles(3, 256, 5), dtype, src_off=src_off, dst_off=dst_off)


@pytest.mark.parametrize("pixels", [16, 64, 256, 1024, 4096, 16384])
def test_fp8_special_values(pixels):
    """Signed zeros, subnormals, NaN and scales outside the range of the corrected quotient (2^-60 to 2^60)."""
    x = tiles(8, pixels, pixels)
    x[1] *= np.float32(1e-24)
    x[2] *= np.float32(1e22)
    x[3] *= np.float32(1e-36)
    x[:, 1::3] = 0.0
    x[:, 2::5] = -0.0
    x[:, 3, 1] = 1e-42
    x[:, 3, 2] = -1e-38
    x[5, 7, 0] = np.nan
    x[6, 7, 1] = -np.float32(np.nan)
    amax = np.nanmax(np.abs(x.reshape(8, -1)), axis=1)
    want = np.where(amax > 0, (amax / np.float32(448.0)).astype(np.float32), np.float32(1.0))
    got, scales = convert(x, D.DFB_FP8E4M3)
    np.testing.assert_array_equal(scales, want)
    q = (x / want[:, None, None]).astype(np.float32)
    np.testing.assert_array_equal(got.reshape(x.shape), o.fp8_e4m3_encode(q.astype(np.float64)))
