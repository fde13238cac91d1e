"""The fixed-order reductions of the split partials, at the edges of their
column groups: rows of whole and of partial 4-column groups, padded and
unaligned rows of Y, odd numbers of partials, fewer and more column groups
than threads of a block, a last block of few rows.  Against the FP64 oracle
with the bound of the arithmetic form (1e-5)."""
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

G, R, U = 0, 1, 2
FP32, BF16 = 0, 1
TOL = 1e-5


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


def _run(P, orc, side, prec, k, m, n, ldy):
    from paper_2603_20966_gb300.workloads import gaussian_matrix
    A = gaussian_matrix(m, n, k + m + n)
    lda = n if prec == FP32 else (n + 3) // 4 * 4
    Ad = torch.zeros((m, lda), device="cuda")
    Ad[:, :n] = A.cuda()
    rows, cols = (k, n) if side == "left" else (m, k)
    Y = torch.full((rows, ldy), float("nan"), device="cuda")
    h = P.sk_create(5, R, k)
    try:
        P.sk_set_precision(h, prec)
        (P.sk_apply_left if side == "left" else P.sk_apply_right)(h, Ad, m, n, lda, Y, ldy)
        assert P.sk_stream_status(h) == 0
    finally:
        P.sk_destroy(h)
    ref = (orc.apply_left if side == "left" else orc.apply_right)(5, R, prec, k, A.numpy())
    assert torch.isnan(Y[:, cols:]).all()
    assert rel_frob(Y[:, :cols].cpu().numpy(), ref) <= TOL


# 16-byte groups (k n / 4 above one block per SM), then the same with a row
# stride or a length that rules them out, then small outputs of many splits
@pytest.mark.parametrize("k,m,n,ldy", [(400, 2000, 400, 400), (400, 2000, 400, 404),
                                       (400, 2000, 400, 401), (401, 2000, 399, 399),
                                       (3, 4100, 5, 5), (1, 9000, 1, 1)])
def test_split_partials(P, orc, k, m, n, ldy):
    _run(P, orc, "left", FP32, k, m, n, ldy)


@pytest.mark.parametrize("k,m,n,ldy", [(100, 1025, 700, 100), (1100, 1030, 300, 1104),
                                       (5, 2100, 900, 8), (258, 40, 500, 260)])
def test_block_segments(P, orc, k, m, n, ldy):
    _run(P, orc, "right", BF16, k, m, n, ldy)
