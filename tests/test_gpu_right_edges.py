"""The BF16 right sketch at the edges of its stages (32 columns of n), its
accumulation chains (2048 columns), its 8-row groups of S and its padded
partial rows, and a lent workspace that has no room for the padding.  Against
the FP64 oracle with the form's bound (1e-5)."""
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

G, R, U = 0, 1, 2
BF16 = 1
TOL = 1e-5


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


def _right(P, dist, k, A, lend=None):
    m, n = A.shape
    lda, ldy = (n + 3) // 4 * 4, (k + 3) // 4 * 4
    Ad = torch.zeros((m, lda), device="cuda")
    Ad[:, :n] = A.cuda()
    Y = torch.full((m, ldy), float("nan"), device="cuda")
    h = P.sk_create(9, dist, k)
    try:
        P.sk_set_precision(h, BF16)
        if lend is not None:
            P.sk_set_workspace(h, lend, lend.numel() * 4)
        P.sk_apply_right(h, Ad, m, n, lda, Y, ldy)
        assert P.sk_stream_status(h) == 0
    finally:
        P.sk_destroy(h)
    assert torch.isnan(Y[:, k:]).all()
    return Y[:, :k].cpu().numpy()


@pytest.mark.parametrize("dist", [G, R, U])
@pytest.mark.parametrize("k,m,n", [(1, 1, 1), (8, 300, 31), (33, 257, 33), (64, 1024, 64),
                                   (97, 1025, 65), (256, 40, 2048), (130, 600, 2081),
                                   (290, 2500, 70)])
def test_right_edges(P, orc, dist, k, m, n):
    from paper_2603_20966_gb300.workloads import gaussian_matrix
    A = gaussian_matrix(m, n, k + m + n)
    assert rel_frob(_right(P, dist, k, A), orc.apply_right(9, dist, BF16, k, A.numpy())) <= TOL


def test_right_without_room_for_padded_rows(P):
    # rows of 167 columns: the largest number of partials is a function of the
    # shape; what is lent holds them with bare rows only
    from paper_2603_20966_gb300.workloads import gaussian_matrix
    k, m, n = 167, 2617, 345
    A = gaussian_matrix(m, n, 3)
    h = P.sk_create(9, G, k)
    P.sk_set_precision(h, BF16)
    padded = P.sk_workspace_size(h, 1, m, n)
    P.sk_destroy(h)
    assert padded % (168 * m * 4) == 0
    bare = padded // 168 * 167
    lend = torch.empty(bare // 4, device="cuda")
    assert (_right(P, G, k, A, lend) == _right(P, G, k, A)).all()
