"""The folded contraction with a tile's K range split between the CTAs of a cluster (gemm_fold.cu): one to eight parts, parts
of unequal length, a last stage of one word, ragged rows and columns, both tile widths, sub-word activation groups, scales
stored as bf16 -- against the oracle, and the same bits from run to run."""
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [
    # M, N, K, beta_a, beta_w, scale dtype
    (49, 100, 352, 32, 32, 0),        # six stages, the last of one word: three parts
    (9, 64, 320, 32, 32, 0),          # five stages: not split
    (128, 128, 1024, 64, 64, 0),      # eight parts of two stages
    (129, 130, 1088, 32, 32, 0),      # four tiles, 17 stages in eight unequal parts
    (10, 33, 4608, 32, 32, 1),        # narrow tile, bf16 scales
    (300, 700, 960, 32, 64, 0),       # 18 tiles: as many CTAs per tile as fit
    (1100, 1000, 512, 32, 32, 0),     # 72 tiles: pairs of CTAs
    (200, 72, 1152, 16, 16, 0),
    (130, 200, 2304, 4, 4, 0),        # scales through the shared-memory ring
    (70, 60, 1088, 2, 16, 0),         # 544 scales per row: row maxima from their own kernel
    (70, 150, 768, 8, 8, 1),
    (40, 50, 640, 640, 32, 0),        # one activation group per row
]


@pytest.mark.parametrize("M,N,K,ba,bw,sdt", CASES)
def test_split_tiles_match_oracle(M, N, K, ba, bw, sdt):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    a, w = inputs.normal((M, K), 4400 + M + K + ba), inputs.he_normal(N, K, 5400 + N + K + bw)
    A, da, sa = gu.oracle_operand(a, ba, sdt)
    W, dw, sw = gu.oracle_operand(w, bw, sdt)
    ea, ew = gu.eff_beta(ba, K), gu.eff_beta(bw, K)
    c_ref, absref = oracle.hbmm_from_quantized(da, sa, ea, dw, sw, ew)
    fine = gu.elementwise_magnitude(da, ea, dw, ew, K)
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    ldc = (N + 3) // 4 * 4 + 4
    outs = [torch.full((M, ldc), float("nan"), device="cuda") for _ in range(3)]
    for C, path in zip(outs, (hbmm.PATH_FOLDED, hbmm.PATH_FOLDED_PREPARED, hbmm.PATH_FOLDED_PREPARED)):
        hbmm.gemm_ex(A, W, C, path, ws)
        assert torch.isnan(C[:, N:]).all()
        assert torch.equal(C[:, :N], outs[0][:, :N])
    gu.assert_close_rel_absref(outs[0][:, :N].cpu().numpy(), c_ref, absref, 1e-5, "split", fine)
    assert hbmm.last_device_error() == 0


@pytest.mark.parametrize("M,N,K,ba,bw", [
    (1300, 1030, 1248, 32, 32),       # 20 stages, 99 tiles: wide accumulator under the balanced schedule
    (1300, 1030, 1216, 32, 32),       # 19: two narrow ones
    (2500, 1000, 1312, 16, 16),       # 160 tiles, whole ones, the last stage of one word
    (2400, 1001, 1280, 8, 8),
])
def test_long_tiles_match_oracle(M, N, K, ba, bw):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    a, w = inputs.normal((M, K), 4500 + M + K + ba), inputs.he_normal(N, K, 5500 + N + K + bw)
    A, da, sa = gu.oracle_operand(a, ba, 0)
    W, dw, sw = gu.oracle_operand(w, bw, 0)
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    C = torch.full((M, (N + 3) // 4 * 4 + 4), float("nan"), device="cuda")
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED, ws)
    assert torch.isnan(C[:, N:]).all()
    rows = list(range(0, M, 97)) + [M - 1]
    c_ref, absref = oracle.hbmm_from_quantized(da[rows], sa[rows], ba, dw, sw, bw)
    fine = gu.elementwise_magnitude(da[rows], ba, dw, bw, K)
    gu.assert_close_rel_absref(C[rows, :N].cpu().numpy(), c_ref, absref, 1e-5, "long tiles", fine)
    # all the other rows: the same product without a workspace, which the oracle holds to 1e-5 as well
    P = torch.empty_like(C)
    hbmm.gemm_ex(A, W, P, hbmm.PATH_POPC)
    diff = (C[:, :N] - P[:, :N]).double()
    assert float(diff.norm() / P[:, :N].double().norm()) < 1e-5


@pytest.mark.parametrize("M,N,K,ba,bw,sdt", [
    (2900, 1001, 256, 32, 32, 0),     # 184 tiles of four stages
    (4000, 700, 288, 32, 16, 1),      # 192 tiles, the last stage of one word, bf16 scales
    (5000, 900, 224, 224, 32, 0),     # 320 tiles: three turns, one activation group per row
    (2560, 1030, 928, 32, 32, 0),     # 15 stages: the longest taken whole at 180 tiles
    (2560, 1030, 1024, 64, 32, 0),    # 16: the balanced schedule
])
def test_short_whole_tiles_match_oracle(M, N, K, ba, bw, sdt):
    """Short 128-column tiles that are walked whole with the wide accumulator, and the first that are not."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    a, w = inputs.normal((M, K), 4600 + M + K + ba), inputs.he_normal(N, K, 5600 + N + K + bw)
    A, da, sa = gu.oracle_operand(a, ba, sdt)
    W, dw, sw = gu.oracle_operand(w, bw, sdt)
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    C = torch.full((M, (N + 3) // 4 * 4 + 4), float("nan"), device="cuda")
    D = torch.full_like(C, float("nan"))
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED, ws)
    hbmm.gemm_ex(A, W, D, hbmm.PATH_FOLDED_PREPARED, ws)
    assert torch.isnan(C[:, N:]).all() and torch.isnan(D[:, N:]).all() and torch.equal(C[:, :N], D[:, :N])
    rows = list(range(0, M, 97)) + [M - 1]
    ea, ew = gu.eff_beta(ba, K), gu.eff_beta(bw, K)
    c_ref, absref = oracle.hbmm_from_quantized(da[rows], sa[rows], ea, dw, sw, ew)
    fine = gu.elementwise_magnitude(da[rows], ea, dw, ew, K)
    gu.assert_close_rel_absref(C[rows, :N].cpu().numpy(), c_ref, absref, 1e-5, "short whole tiles", fine)
    hbmm.gemm_ex(A, W, D, hbmm.PATH_POPC)      # all the other rows: without a workspace, which the oracle holds to 1e-5 as well
    assert float((C - D)[:, :N].double().norm() / D[:, :N].double().norm()) < 1e-5


def test_row_pitch_that_no_tensor_copy_takes():
    """One row whose pitch (2^38 elements) is beyond a tensor copy's: the blocks leave by plain stores, with the same values."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    N, K = 103, 256
    A, _, _ = gu.oracle_operand(inputs.normal((1, K), 4700), 32, 0)
    W, _, _ = gu.oracle_operand(inputs.he_normal(N, K, 5700), 32, 0)
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    C, D = torch.full((1, 108), float("nan"), device="cuda"), torch.full((1, 108), float("nan"), device="cuda")
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED, ws)
    hbmm.gemm_ex(A, W, D.as_strided((1, 108), (1 << 38, 1)), hbmm.PATH_FOLDED_PREPARED, ws)
    assert torch.equal(C[:, :N], D[:, :N]) and torch.isnan(C[:, N:]).all() and torch.isnan(D[:, N:]).all()


def test_tiles_walked_in_blocks_of_columns():
    """More expanded weights than the L2 keeps: every tile is still formed once (blocks of 11 columns, a last one of 10; row
    and column remainders).  Against the workspace-free tiles, which the oracle holds to 1e-5 elsewhere."""
    from paper_1905_10759_b200 import hbmm
    M, N, K, b = 2500, 4090, 3200, 32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x, w = (torch.randn((r, K), generator=gen, device="cuda") for r in (M, N))
    A, W = hbmm.quantize(x, hbmm.alloc_operand(M, K, b)), hbmm.quantize(w, hbmm.alloc_operand(N, K, b))
    ws = torch.empty(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    C = torch.full((M, 4096), float("nan"), device="cuda")
    P = torch.empty_like(C)
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED, ws)
    hbmm.gemm_ex(A, W, P, hbmm.PATH_POPC)
    assert torch.isnan(C[:, N:]).all()
    diff, ref = (C[:, :N] - P[:, :N]).double(), P[:, :N].double()
    assert float(diff.norm() / ref.norm()) < 1e-5
    assert float(diff.abs().max()) < 1e-3 * float(ref.abs().max())


def test_prepared_calls_with_any_number_of_rows():
    """One expansion serves calls of 10 to 1040 tiles in any order, split, balanced and plain, in a workspace that held
    something else before: the same bits as a call that expands the weights itself."""
    from paper_1905_10759_b200 import hbmm
    N, K, b = 1280, 1024, 64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(11)
    W = hbmm.quantize(torch.randn((N, K), generator=gen, device="cuda"), hbmm.alloc_operand(N, K, b))
    ops = {M: hbmm.quantize(torch.randn((M, K), generator=gen, device="cuda"), hbmm.alloc_operand(M, K, b))
           for M in (128, 1024, 1408, 13200)}
    nbytes = max(hbmm.gemm_workspace_bytes(A, W) for A in ops.values())

    def product(M, path, ws):
        C = torch.full((M, N), float("nan"), device="cuda")
        hbmm.gemm_ex(ops[M], W, C, path, ws)
        return C

    junk = lambda: torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")
    fresh = {M: product(M, hbmm.PATH_FOLDED, junk()) for M in ops}
    for first in (128, 1408, 13200):
        ws = junk()
        assert torch.equal(product(first, hbmm.PATH_FOLDED, ws), fresh[first])
        for M in (1408, 1024, 1408, 128, 13200, 1024):
            assert torch.equal(product(M, hbmm.PATH_FOLDED_PREPARED, ws), fresh[M]), (first, M)
