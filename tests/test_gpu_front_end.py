"""Packed convolution front end on strided filters (tensor-copy tiles of fewer rows, whole channel planes), on the gather for
groups shorter than a word (bf16 images, odd widths, large filters, K ending inside a word; 3 x 3 at stride 1 and 1 x 1 have
kernels of their own) and on the staged tiles of 3 x 3 filters that are not walked: the packed operand left in the workspace
against the oracle's binarization of the im2col rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, H, W, k, stride, beta, bf16
    (2, 64, 56, 56, 3, 2, 32, False),     # two tiles fit only with fewer output rows
    (3, 40, 28, 28, 3, 2, 64, False),     # short last channel chunk, groups of two words
    (2, 64, 14, 14, 3, 2, 32, False),     # whole planes
    (2, 32, 13, 16, 3, 2, 8, False),
    (2, 64, 8, 8, 1, 2, 4, False),
    (1, 32, 60, 60, 5, 3, 32, False),
    (2, 100, 9, 9, 3, 1, 16, False),      # odd width, K = 900
    (2, 33, 7, 7, 5, 1, 2, False),        # K = 825
    (2, 48, 12, 12, 3, 2, 4, True),       # bf16 image
    (1, 5, 11, 10, 3, 1, 8, True),        # K = 45: two words, a short group
    (1, 3, 11, 10, 5, 1, 8, True),        # K = 75: three words, a short group
]


@pytest.mark.parametrize("B,C,H,W,k,st,beta,bf16", CASES)
def test_packed_rows_match_oracle(B, C, H, W, k, st, beta, bf16):
    packed_rows(B, C, H, W, k, (st, st), k // 2, beta, bf16)


@pytest.mark.parametrize("B,C,H,W,sh,pad,bf16", [
    (2, 64, 9, 13, 2, 1, True),           # stride over the rows only
    (1, 40, 7, 10, 1, 3, True),           # wide padding, short last channel chunk
    (1, 33, 11, 6, 2, 0, False),          # a chunk of one channel
])
def test_tiles_with_constant_offsets_match_oracle(B, C, H, W, sh, pad, bf16):
    """3 x 3 filters at beta 32 that neither the walked columns nor the tensor copies take."""
    packed_rows(B, C, H, W, 3, (sh, 1), pad, 32, bf16)


def packed_rows(B, C, H, W, k, st, pad, beta, bf16):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    K = C * k * k
    x = inputs.normal((B * C * H, W), 650 + C + H).reshape(B, C, H, W)
    if bf16:
        x = torch.from_numpy(x).bfloat16().float().numpy()
    Wop = hbmm.quantize(torch.from_numpy(inputs.he_normal(40, K, 651)).cuda(), hbmm.alloc_operand(40, K, max(beta, 32)))
    geom = hbmm.make_geom(B, C, H, W, k, k, st, (pad, pad))
    M = B * ((H + 2 * pad - k) // st[0] + 1) * ((W + 2 * pad - k) // st[1] + 1)
    ws = torch.empty(hbmm.conv_workspace_bytes(geom, beta, hbmm.F32, Wop), dtype=torch.uint8, device="cuda").fill_(0xAB)
    xd = torch.from_numpy(x).cuda()
    hbmm.conv_im2col(xd.bfloat16() if bf16 else xd, geom, beta, hbmm.F32, Wop, None, ws, flags=hbmm.CONV_PACK_ONLY)
    bb, sb, lw, ls = hbmm.operand_bytes(M, K, beta, hbmm.F32)
    bits = ws[:bb].view(torch.int32).reshape(M, lw)
    off = (bb + 255) // 256 * 256
    sc = ws[off: off + sb].view(torch.float32).reshape(M, ls).cpu().numpy().astype(np.float64)
    da, sa = oracle.quantize(oracle.im2col(x, k, k, st, (pad, pad)), beta)
    assert np.array_equal(gu.host_bits(bits), oracle.pack(sa, lw))
    G = da.shape[1]
    assert np.all(sc[:, G:] == 0.0)
    # four partial sums of a word's or group's elements in turn, joined pairwise, one division
    np.testing.assert_allclose(sc[:, :G], da, rtol=(min(beta, 32) // 4 + int(np.ceil(np.log2(beta))) + 3) * gu.U, atol=0)
    assert hbmm.last_device_error() == 0


@pytest.mark.parametrize("first", ["bf16", "off by one element"])
@pytest.mark.parametrize("beta", [8, 16, 32, 64])
@pytest.mark.parametrize("B,H,Wd,st", [(2, 4, 4, 1), (1, 5, 8, 2)])
def test_weights_of_a_first_call_serve_the_other_front_end(B, H, Wd, st, beta, first):
    """At most eight output pixels.  At stride 2 the first call's image takes the gathering front end, the prepared calls' (plain
    and fused) the tensor-copy one; at stride 1 both are walked, from images of another type or alignment.  The workspace held
    something else before."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    C, N = 32, 40
    K, M = C * 9, B * ((H - 3) // st + 1) * ((Wd - 3) // st + 1)
    x = inputs.normal((B * C * H, Wd), 6100 + beta).reshape(B, C, H, Wd)
    w = inputs.he_normal(N, K, 6200 + beta)
    W = hbmm.quantize(torch.from_numpy(w).cuda(), hbmm.alloc_operand(N, K, beta))
    geom = hbmm.make_geom(B, C, H, Wd, 3, 3, (st, st))
    ws = torch.full((hbmm.conv_workspace_bytes(geom, beta, hbmm.F32, W),), 0xFF, dtype=torch.uint8, device="cuda")
    xd = torch.from_numpy(x).cuda()
    if first == "bf16":
        x1 = xd.bfloat16()
    else:
        x1 = torch.empty(xd.numel() + 1, device="cuda")[1:].view(xd.shape).copy_(xd)
    out = torch.full((M, N), float("nan"), device="cuda")
    hbmm.conv_im2col(x1, geom, beta, hbmm.F32, W, torch.empty((M, N), device="cuda"), ws)
    hbmm.conv_im2col(xd, geom, beta, hbmm.F32, W, out, ws, flags=hbmm.CONV_WEIGHTS_PREPARED)
    c_ref, absref = oracle.conv_im2col(x, w, 3, 3, (st, st), (0, 0), beta, beta)
    da, dw = oracle.quantize(oracle.im2col(x, 3, 3, (st, st)), beta)[0], oracle.quantize(w, beta)[0]
    fine = gu.elementwise_magnitude(da, beta, dw, beta, K)
    gu.assert_close_rel_absref(out.cpu().numpy(), c_ref, absref, 1e-5, "prepared", fine)
    if beta >= 32:
        z = torch.full((M, N), float("nan"), device="cuda")
        hbmm.conv_im2col_fused(xd, geom, beta, hbmm.F32, W, hbmm.make_epilogue(out=z), ws, flags=hbmm.CONV_WEIGHTS_PREPARED)
        gu.assert_close_rel_absref(z.cpu().numpy(), c_ref, absref, 1e-5, "fused, prepared", fine)
