"""Packed convolution front ends of 3 x 3 filters at stride 1 (columns walked down the image) and of 1 x 1 filters: the packed
operand left in the workspace against the oracle's binarization of the im2col rows, at the edges of their lanes, strips, row
segments, channel pieces and ranges."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, H, W, pad, beta, bf16 image, bf16 scales
    (2, 64, 9, 30, 1, 32, False, False),   # a strip of 30 columns fills the warp's lanes
    (1, 64, 9, 31, 1, 32, True, False),    # ... one column more takes two strips
    (3, 32, 5, 7, 1, 16, False, True),     # three strips of a warp, the last rows of a segment missing
    (1, 288, 4, 3, 1, 64, False, False),   # three channel ranges, the last of one chunk; one column
    (2, 136, 6, 14, 1, 8, False, False),   # ranges that start between 16-byte pieces of words
    (2, 44, 6, 14, 1, 4, True, True),      # a piece of four channels ends the row inside a byte
    (1, 33, 8, 9, 2, 2, False, False),     # a piece of one channel; two columns of padding
    (2, 5, 3, 3, 0, 32, False, False),     # one output pixel, K = 45
    (1, 256, 13, 13, 1, 256, False, True), # a group of eight words spans four chunks
    (1, 96, 3, 90, 1, 96, True, False),    # groups of three words
    (5, 20, 2, 1, 1, 16, False, False),    # one input column
    (2, 8, 6, 9, 1, 32, False, False),     # images of fewer channels than a lane holds: all of 8,
    (1, 7, 5, 8, 1, 16, True, False),      # ... 7 of 8,
    (2, 16, 6, 9, 1, 32, True, True),      # 16,
    (1, 9, 5, 7, 2, 64, False, False),     # 9 of 16, a short group of two words,
    (2, 24, 6, 9, 1, 96, False, False),    # 24,
    (1, 17, 9, 9, 1, 32, False, False),    # 17 of 24
    (2, 3, 7, 7, 1, 16, False, False),
    (1, 3, 5, 5, 0, 16, False, True),      # K = 27: a short second group
    (2, 25, 6, 9, 1, 32, False, False),    # ... and one channel more: all 32
    (1, 130, 6, 9, 1, 16, False, False),   # two channel ranges at beta 16, the last of two channels
]


POINT_CASES = [
    # the same for 1 x 1 filters, with their stride
    (2, 64, 9, 31, 1, 0, 32, False, False),
    (1, 100, 7, 13, 2, 0, 4, True, True),     # the last word of four channels
    (3, 48, 5, 5, 2, 1, 16, False, False),    # padding: rows of zeros
    (1, 33, 3, 3, 1, 0, 8, False, False),
    (1, 70, 8, 8, 3, 0, 2, True, False),
    (2, 260, 6, 6, 1, 0, 64, False, True),    # a last group of four channels
    (1, 512, 4, 4, 1, 0, 256, False, False),
    (2, 64, 6, 6, 1, 0, 64, True, False),     # one group per row
    (2, 10, 6, 6, 1, 0, 16, False, False),
    (2, 3, 7, 7, 1, 1, 96, True, True),       # rows of one word and one group, stored whole
    (2, 8, 7, 7, 1, 0, 2, True, False),       # all of eight channels, one of them, one more
    (1, 2, 6, 7, 1, 0, 16, False, False),
    (1, 9, 6, 7, 1, 1, 4, False, False),
    (1, 32, 9, 15, 2, 0, 32, False, False),
    (3, 31, 5, 5, 1, 0, 4, False, True),
]


@pytest.mark.parametrize("B,C,H,W,pad,beta,bf16,sbf16", CASES)
def test_packed_rows_match_oracle(B, C, H, W, pad, beta, bf16, sbf16):
    packed_rows(B, C, H, W, 3, 1, pad, beta, bf16, sbf16)


@pytest.mark.parametrize("B,C,H,W,st,pad,beta,bf16,sbf16", POINT_CASES)
def test_packed_pixels_match_oracle(B, C, H, W, st, pad, beta, bf16, sbf16):
    packed_rows(B, C, H, W, 1, st, pad, beta, bf16, sbf16)


def packed_rows(B, C, H, W, k, st, pad, beta, bf16, sbf16):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    K = C * k * k
    x = inputs.normal((B * C * H, W), 760 + C + W).reshape(B, C, H, W).copy()
    x.reshape(-1)[::7] = 0.0
    x.reshape(-1)[::11] = -0.0
    if bf16:
        x = torch.from_numpy(x).bfloat16().float().numpy()
    sdt = hbmm.BF16 if sbf16 else hbmm.F32
    Wop = hbmm.quantize(torch.from_numpy(inputs.he_normal(40, K, 761)).cuda(), hbmm.alloc_operand(40, K, max(beta, 32)))
    geom = hbmm.make_geom(B, C, H, W, k, k, (st, st), (pad, pad))
    M = B * ((H + 2 * pad - k) // st + 1) * ((W + 2 * pad - k) // st + 1)
    ws = torch.empty(hbmm.conv_workspace_bytes(geom, beta, sdt, Wop), dtype=torch.uint8, device="cuda").fill_(0xAB)
    # an image off any vector's alignment: only the element's own is asked for
    xd = torch.empty(x.size + 1, dtype=torch.bfloat16 if bf16 else torch.float32, device="cuda")[1:].view(x.shape).copy_(torch.from_numpy(x))
    hbmm.conv_im2col(xd, geom, beta, sdt, Wop, None, ws, flags=hbmm.CONV_PACK_ONLY)
    bb, sb, lw, ls = hbmm.operand_bytes(M, K, beta, sdt)
    bits = ws[:bb].view(torch.int32).reshape(M, lw)
    off = (bb + 255) // 256 * 256
    sc = ws[off: off + sb].view(torch.bfloat16 if sbf16 else torch.float32).reshape(M, ls).float().cpu().numpy().astype(np.float64)
    da, sa = oracle.quantize(oracle.im2col(x, k, k, (st, st), (pad, pad)), gu.eff_beta(beta, K))
    assert np.array_equal(gu.host_bits(bits), oracle.pack(sa, lw))
    G = da.shape[1]
    assert np.all(sc[:, G:] == 0.0)
    # a word's elements: up to three channels, two neighbours, a cut channel's part and two rows added (eight additions deep),
    # the words of a group in turn, one division; half a unit of eight bits more for bf16 scales
    np.testing.assert_allclose(sc[:, :G], da, rtol=(8 + beta // 32 + 1) * gu.U + (2.0 ** -8 if sbf16 else 0.0), atol=0)
    assert hbmm.last_device_error() == 0
