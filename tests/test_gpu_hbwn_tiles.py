"""Dense-activation convolution: the 64-column tiles of CTA pairs and the epilogue that leaves by tensor copies, at the sizes
where they can go wrong -- one row tile, row and column remainders, column counts that end inside 16 bytes, output rows off 16
bytes, two turns of tiles, packed groups as wide as the wide tile -- against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    # B, C, H, N, kind of output, pitch beyond N
    (1, 64, 7, 65, "product", 3),         # 49 rows, one column in the second tile
    (3, 64, 14, 192, "product", 0),       # three tiles of 64 on two of the prepared 128
    (5, 64, 14, 98, "product", 2),        # the last block ends inside four columns
    (2, 128, 14, 100, "bf16", 0),         # ... and inside eight
    (2, 64, 14, 136, "bf16", 0),
    (2, 64, 14, 130, "fp32", 2),
    (2, 64, 9, 72, "bf16", 3),            # rows off 16 bytes
    (1, 64, 9, 96, "packed 32", 0),
    (3, 64, 9, 200, "packed 64", 0),
    (3, 64, 9, 200, "packed 128", 0),     # a group fills the wide tile
    (16, 64, 24, 256, "bf16", 0),         # more narrow tiles than pairs
]


@pytest.mark.parametrize("B,C,H,N,kind,extra", CASES)
def test_tiles_match_oracle(B, C, H, N, kind, extra):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    K, M, beta = C * 9, B * H * H, 32
    x = torch.from_numpy(inputs.normal((B * C * H, H), 8100 + N).reshape(B, C, H, H)).bfloat16()
    w = inputs.he_normal(N, K, 8200 + N)
    W = hbmm.quantize(torch.from_numpy(w).cuda(), hbmm.alloc_operand(N, K, beta))
    geom = hbmm.make_geom(B, C, H, H, 3, 3, (1, 1), (1, 1))
    ws = torch.empty(hbmm.conv_workspace_bytes(geom, 1, hbmm.F32, W), dtype=torch.uint8, device="cuda").fill_(0xFF)
    xd = x.cuda()
    c_ref, absref = oracle.conv_im2col(x.float().numpy(), w, 3, 3, (1, 1), (1, 1), 1, beta)
    # two bf16 pieces per weight (2^-18), fp32 sums of K terms in the tensor core
    tol = ((beta + K // beta + 4) * 2 * gu.U + 2.0 ** -18) * absref + 1e-12 * max(1.0, absref.max())
    if kind == "product":
        out = torch.full((M, (N + 3) // 4 * 4 + 4 * extra), float("nan"), device="cuda")
        hbmm.conv_im2col(xd, geom, 1, hbmm.F32, W, out, ws)
        assert torch.isnan(out[:, N:]).all()
        assert (np.abs(out[:, :N].cpu().numpy().astype(np.float64) - c_ref) <= tol).all()
        return
    sc, sh = np.abs(inputs.normal((N,), 8300)) + 0.5, inputs.normal((N,), 8301)
    args = (hbmm.ACT_RELU, torch.from_numpy(sc).cuda(), torch.from_numpy(sh).cuda())
    z, band = np.maximum(c_ref, 0.0) * sc + sh, tol * sc + 4 * gu.U * (np.abs(c_ref * sc) + np.abs(sh))
    if kind.startswith("packed"):
        bn = int(kind.split()[1])
        nxt = hbmm.alloc_operand(M, N, bn)
        nxt.bits.fill_(-1)
        nxt.scales.fill_(float("nan"))
        hbmm.conv_im2col_fused(xd, geom, 1, hbmm.F32, W, hbmm.make_epilogue(*args, nxt=nxt), ws)
        da, sa = oracle.quantize(z.astype(np.float32), bn)
        words = gu.host_bits(nxt.bits)
        got = ((words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1).reshape(M, -1)
        clear = np.abs(z) > band
        assert (got[:, :N][clear] == (z >= 0)[clear]).all() and clear.mean() > 0.99
        assert not got[:, N:].any()
        G = da.shape[1]
        s = nxt.scales.cpu().numpy().astype(np.float64)
        edge = np.pad(band, ((0, 0), (0, G * bn - N))).reshape(M, G, bn).sum(2) / np.minimum(bn, N - np.arange(G) * bn)
        assert (np.abs(s[:, :G] - da) <= edge + (np.log2(bn) + 3) * gu.U * da).all() and not s[:, G:].any()
        return
    dt = torch.bfloat16 if kind == "bf16" else torch.float32
    out = torch.full((M, N + extra), 7.0, dtype=dt, device="cuda")
    hbmm.conv_im2col_fused(xd, geom, 1, hbmm.F32, W, hbmm.make_epilogue(*args, out=out[:, :N]), ws)
    assert (out[:, N:] == 7.0).all()
    got = out[:, :N].float().cpu().numpy().astype(np.float64)
    assert (np.abs(got - z) <= band + (2.0 ** -8 * np.abs(z) if kind == "bf16" else 0.0) + 1e-12).all()


@pytest.mark.parametrize("M,N", [(1, 1024), (1, 1025), (3, 1100), (4, 1025), (5, 2048), (5, 2049), (63, 2100), (64, 2100)])
def test_few_rows_match_oracle(M, N):
    """One row tile, at the limits of rows and columns between narrow tiles of CTA pairs and one CTA per 128 columns."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    K, beta = 128, 32
    a = torch.from_numpy(inputs.normal((M, K), 8400 + N)).bfloat16()
    w = inputs.he_normal(N, K, 8500 + N)
    A, W = hbmm.wrap_dense(a.cuda()), hbmm.quantize(torch.from_numpy(w).cuda(), hbmm.alloc_operand(N, K, beta))
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda").fill_(0xFF)
    C = torch.full((M, (N + 3) // 4 * 4 + 4), float("nan"), device="cuda")
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED, ws)
    dw, sw = oracle.quantize(w, beta)
    wb = np.repeat(dw, beta, axis=1)[:, :K] * sw
    x = a.float().numpy().astype(np.float64)
    tol = (K + 4) * gu.U * (np.abs(x) @ np.abs(wb).T) + 2.0 ** -18 * (np.abs(x) @ np.abs(wb).T)
    assert (np.abs(C[:, :N].cpu().numpy() - x @ wb.T) <= tol).all() and torch.isnan(C[:, N:]).all()
    assert hbmm.last_device_error() == 0
