"""Streams over rows that end inside a group (backward.cu, binarize_dense.cu): every group size, row lengths around the 128
elements a warp takes, row starts on and off 16-byte boundaries -- against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [(r, K, b, pad) for b in (1, 2, 4, 8, 16, 32, 64, 128) for r, K, pad in ((9, 131, 0), (5, 260, 4), (3, 388 - b // 2, 1))]
CASES += [(7, 64, 128, 0), (1, 65, 64, 3), (300, 127, 16, 0)]
CASES += [(9, 126, 4, 0), (5, 250, 4, 6), (3, 511, 4, 1)]          # nearly full warps: groups of four take them only then


@pytest.mark.parametrize("rows,K,beta,pad", CASES)
def test_row_streams_match_oracle(rows, K, beta, pad):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    x, gy = inputs.normal((rows, K), 9400 + rows + K), inputs.normal((rows, K), 9500 + rows + beta)
    x[0, :4] = [1.0, -1.0, 0.0, -0.0]
    xd, gd = torch.zeros((rows, K + pad)), torch.zeros((rows, K + pad))
    xd[:, :K], gd[:, :K] = torch.from_numpy(x), torch.from_numpy(gy)
    xg, gg = xd.cuda()[:, :K], gd.cuda()[:, :K]
    be = gu.eff_beta(beta, K)
    delta, sign = oracle.quantize(x, be)
    ref = oracle.dequant(delta, sign, be)
    out = torch.full((rows, K + pad), float("nan"), device="cuda")
    hbmm.binarize_dense(xg, beta, hbmm.F32, out[:, :K])
    got = out.cpu().numpy()
    assert np.isnan(got[:, K:]).all()
    got = got[:, :K]
    assert np.array_equal(np.signbit(got), sign < 0)
    # an fp32 tree over the group and one division
    tree = int(np.ceil(np.log2(max(be, 2)))) + int(np.ceil(be / 32))
    assert (np.abs(np.abs(got.astype(np.float64)) - np.abs(ref)) <= (tree + 2) * gu.U * np.abs(ref)).all()
    outb = torch.full((rows, K + pad), float("nan"), device="cuda", dtype=torch.bfloat16)
    hbmm.binarize_dense(xg, beta, hbmm.BF16, outb[:, :K])
    assert torch.isnan(outb[:, K:]).all()
    assert torch.equal(outb[:, :K], out[:, :K].to(torch.bfloat16))
    gx = torch.full((rows, K + pad), float("nan"), device="cuda")
    hbmm.binarize_backward(xg, gg, beta, gx[:, :K])
    got = gx.cpu().numpy()
    assert np.isnan(got[:, K:]).all()
    # two such trees, one division and one multiply each, one add
    x64, g64 = np.abs(x.astype(np.float64)), np.abs(gy.astype(np.float64))
    mag = np.empty_like(x64)
    for k in range(0, K, be):
        sl = slice(k, min(k + be, K))
        mag[:, sl] = g64[:, sl].mean(axis=1, keepdims=True) + x64[:, sl].mean(axis=1, keepdims=True) * g64[:, sl]
    err = np.abs(got[:, :K].astype(np.float64) - oracle.binarize_backward(x, gy, beta))
    assert (err <= (tree + 4) * gu.U * mag + 1e-30).all()
