"""Products of one to eight rows on groups shorter than a word: the matrix-vector kernel (gemv_popc.cu) and, for many rows of
few words, the tiles; K ending inside a word and inside a group, a row shorter than a warp's stride, mixed groups, one group per
row, bf16 scales -- against the oracle.  And what an automatic call on such rows leaves for prepared ones."""
import pytest
import torch

import oracle
from paper_1905_10759_b200 import inputs

pytestmark = pytest.mark.gpu

CASES = [(M, N, K, b, b, 0) for b in (2, 4, 8, 16) for M, N, K in ((1, 9, 31), (3, 33, 1056), (8, 17, 2055))]
CASES += [(6, 21, 301, 16, 16, 0), (5, 30, 1111, 16, 16, 1)]      # five and six rows at 16: beyond, the tiles take them
CASES += [(5, 40, 777, 2, 64, 0), (2, 41, 777, 32, 8, 1), (4, 7, 333, 333, 16, 0), (6, 8, 100, 4, 4, 1), (7, 1500, 96, 16, 2, 0)]


@pytest.mark.parametrize("M,N,K,ba,bw,sdt", CASES)
def test_gemv_of_sub_word_groups_matches_oracle(M, N, K, ba, bw, sdt):
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    a, w = inputs.normal((M, K), 4200 + M + K + ba), inputs.he_normal(N, K, 5200 + N + K + bw)
    A, da, sa = gu.oracle_operand(a, ba, sdt)
    W, dw, sw = gu.oracle_operand(w, bw, sdt)
    ea, ew = gu.eff_beta(ba, K), gu.eff_beta(bw, K)
    c_ref, absref = oracle.hbmm_from_quantized(da, sa, ea, dw, sw, ew)
    T = -(-K // min(ea, ew))
    for path in (hbmm.PATH_POPC, hbmm.PATH_AUTO):
        C = torch.full((M, (N + 3) // 4 * 4 + 4), float("nan"), device="cuda")
        hbmm.gemm_ex(A, W, C, path)
        assert torch.isnan(C[:, N:]).all()
        # two roundings per segment, one per segment of a lane's sum and five in the tree that joins the lanes
        gu.assert_close_rel_absref(C[:, :N].cpu().numpy(), c_ref, absref, (T + 5 + 2) * gu.U, "gemv")


def test_prepared_call_after_an_automatic_one_on_a_few_rows():
    """A prepared call may follow an automatic one on the same few rows."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    M, N, K, b = 4, 40, 320, 8
    a, w = inputs.normal((M, K), 4300), inputs.he_normal(N, K, 5300)
    A, da, sa = gu.oracle_operand(a, b, 0)
    W, dw, sw = gu.oracle_operand(w, b, 0)
    c_ref, absref = oracle.hbmm_from_quantized(da, sa, b, dw, sw, b)
    ws = torch.zeros(hbmm.gemm_workspace_bytes(A, W), dtype=torch.uint8, device="cuda")
    C = torch.full((M, N), float("nan"), device="cuda")
    hbmm.gemm(A, W, C, ws)
    C.fill_(float("nan"))
    hbmm.gemm_ex(A, W, C, hbmm.PATH_FOLDED_PREPARED, ws)
    gu.assert_close_rel_absref(C.cpu().numpy(), c_ref, absref, 1e-5, "prepared")


def _junk(nbytes):
    return torch.full((nbytes,), 0xFF, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("b,sdt", [(2, 0), (4, 1), (8, 0), (16, 1)])
def test_automatic_call_on_a_few_rows_prepares_calls_on_any(b, sdt):
    """What an automatic call on four rows leaves in a workspace that held anything before serves a prepared call on the
    same rows and one on sixty-four; the three ways to the folded kernel give the same bits."""
    import gpu_util as gu
    from paper_1905_10759_b200 import hbmm
    N, K = 40, 320
    W, dw, sw = gu.oracle_operand(inputs.he_normal(N, K, 5300), b, sdt)
    ops = [gu.oracle_operand(inputs.normal((M, K), 4300 + M), b, sdt) for M in (4, 64)]
    ws = _junk(max(hbmm.gemm_workspace_bytes(A, W) for A, _, _ in ops))
    outs = []
    for (A, da, sa), path in ((ops[0], hbmm.PATH_AUTO), (ops[0], hbmm.PATH_FOLDED_PREPARED), (ops[1], hbmm.PATH_FOLDED_PREPARED)):
        C = torch.full((A.rows, N), float("nan"), device="cuda")
        hbmm.gemm_ex(A, W, C, path, ws)
        outs.append(C)
        assert torch.isfinite(C).all(), path
        c_ref, absref = oracle.hbmm_from_quantized(da, sa, b, dw, sw, b)
        gu.assert_close_rel_absref(C.cpu().numpy(), c_ref, absref, 1e-5, "path %d" % path, gu.elementwise_magnitude(da, b, dw, b, K))
    fresh = torch.full((4, N), float("nan"), device="cuda")
    hbmm.gemm_ex(ops[0][0], W, fresh, hbmm.PATH_FOLDED, _junk(ws.numel()))
    assert torch.equal(outs[0], fresh) and torch.equal(outs[1], fresh)
