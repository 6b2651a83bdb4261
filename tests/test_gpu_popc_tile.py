"""The workspace-free contraction in warp tiles (gemm_popc_tile.cu) at the sizes where it can go wrong: edges of the 32 x 32
tile, every segment length, chunks and K ranges that end inside a word, a segment or a warp's share, one group per row,
mixed groups, both scale types -- against the oracle."""
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [(M, N, K, b, b, 0) for b in (2, 4, 8, 16, 32, 64, 128, 256)
         for M, N, K in ((1, 1, 300), (33, 31, 1055), (32, 65, 2048 + b // 2))]
CASES += [
    (9, 40, 31, 2, 2, 0),            # one word: no K range to split
    (70, 33, 1000, 16, 16, 1),       # bf16 scales
    (40, 36, 777, 2, 64, 0),         # a scale per segment against one per 32 segments
    (40, 36, 777, 96, 32, 1),        # three segments per group
    (300, 130, 200, 200, 200, 0),    # one group per row in both: one segment of eight words
    (50, 60, 333, 333, 4, 0),
    (600, 2050, 96, 32, 32, 0),      # enough tiles that one warp walks the whole of K
    (600, 1030, 290, 8, 8, 0),       # two warps per tile
    (600, 2050, 128, 32, 32, 0),     # whole chunks only: one to a warp,
    (33, 70, 1152, 64, 32, 0),       # ... nine in eight parts,
    (40, 37, 640, 128, 128, 1),
    (40, 36, 512, 256, 256, 0),
    (41, 38, 1000, 96, 32, 0),       # whole ones and one that ends inside its last word
]


@pytest.mark.parametrize("M,N,K,ba,bw,sdt", CASES)
def test_popc_tiles_match_oracle(M, N, K, ba, bw, sdt):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    a, w = inputs.normal((M, K), 4100 + M + K + ba), inputs.he_normal(N, K, 5100 + N + K + bw)
    A, da, sa = gu.oracle_operand(a, ba, sdt)
    W, dw, sw = gu.oracle_operand(w, bw, sdt)
    ea, ew = gu.eff_beta(ba, K), gu.eff_beta(bw, K)
    c_ref, absref = oracle.hbmm_from_quantized(da, sa, ea, dw, sw, ew)
    C = torch.full((M, (N + 3) // 4 * 4 + 4), float("nan"), device="cuda")
    hbmm.gemm_ex(A, W, C, hbmm.PATH_POPC)
    out = C.cpu().numpy()
    assert torch.isnan(C[:, N:]).all()
    # per segment two roundings, then at most one per segment and one per joined part
    T = -(-K // min(ea, ew))
    gu.assert_close_rel_absref(out[:, :N], c_ref, absref, (T + 8 + 2) * gu.U, "popc")


@pytest.mark.parametrize("N", [1, 2, 3])
@pytest.mark.parametrize("b", [2, 4, 8, 16, 32, 64, 128, 256])
def test_narrowest_tiles_match_oracle(b, N):
    """Nine rows (the fewest that reach this kernel) and columns that no vector store covers; K of less than one chunk, and
    of several with words past the row's end in the last."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    for K in (21, 1061):
        a, w = inputs.normal((9, K), 4150 + K + b), inputs.he_normal(N, K, 5150 + N + K + b)
        A, da, sa = gu.oracle_operand(a, b, 0)
        W, dw, sw = gu.oracle_operand(w, b, 0)
        e = gu.eff_beta(b, K)
        c_ref, absref = oracle.hbmm_from_quantized(da, sa, e, dw, sw, e)
        C = torch.full((9, 8), float("nan"), device="cuda")
        hbmm.gemm_ex(A, W, C, hbmm.PATH_POPC)
        assert torch.isnan(C[:, N:]).all()
        gu.assert_close_rel_absref(C[:, :N].cpu().numpy(), c_ref, absref, (-(-K // e) + 8 + 2) * gu.U, "popc")


@pytest.mark.parametrize("b", [32, 64, 128, 256])
def test_cancelling_group_with_scales_beyond_the_range_of_their_product(b):
    """A group of whole words whose signs cancel adds nothing, also where the product of its two scales is above the largest fp32."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    import numpy as np
    M, N, K = 40, 33, 4 * b
    a, w = np.ones((M, K), np.float32), np.ones((N, K), np.float32)
    a[:, b: 2 * b], w[:, b: 2 * b] = 1e25, 1e25
    w[:, b: 2 * b: 2] = -1e25
    A, da, sa = gu.oracle_operand(a, b, 0)
    W, dw, sw = gu.oracle_operand(w, b, 0)
    C = torch.full((M, (N + 3) // 4 * 4), float("nan"), device="cuda")
    hbmm.gemm_ex(A, W, C, hbmm.PATH_POPC)
    assert torch.equal(C[:, :N].cpu(), torch.full((M, N), float(3 * b)))
