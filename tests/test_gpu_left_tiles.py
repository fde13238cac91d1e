"""BF16 split-A left sketch on CTA pairs at the rows of the last 256-row tile
of S, which the two CTAs share in whole 32-row boxes: every step of that rule,
drained through the TMA and (rows of a lent workspace without padding) by the
transpose tiles; within 1e-5 of the FP64 oracle, the form's bound."""
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

G, R = 0, 1
TOL = 1e-5


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


@pytest.mark.parametrize("dist", [G, R])
@pytest.mark.parametrize("k", [129, 160, 192, 193, 256, 257, 288, 289, 320, 321, 385, 449, 511])
def test_rows_of_the_last_tile(P, orc, dist, k):
    from paper_2603_20966_gb300.workloads import gaussian_matrix
    m, n = 2100, 97
    A = gaussian_matrix(m, n, k, device="cpu")
    ref = orc.apply_left(7, dist, 1, k, A.numpy())
    Ad = torch.zeros((m, 100), dtype=torch.float32, device="cuda")
    Ad[:, :n] = A.cuda()
    with P.Sketch(7, dist, k, P.SK_BF16X2) as S:
        for lent in (False, True):
            if lent:
                # rows of 97 columns leave too little for padded ones
                size = P.sk_workspace_size(S.handle, 0, m, n)
                ws = torch.empty(size, dtype=torch.uint8, device="cuda")
                small, least = 0, size  # the smallest buffer the call takes
                while least - small > 16:
                    P.sk_set_workspace(S.handle, ws.data_ptr(), (small + least) // 2)
                    try:
                        P.sk_apply_left(S.handle, Ad, m, n, 100,
                                        torch.empty((k, 100), device="cuda"), 100)
                        least = (small + least) // 2
                    except P.SketchError:
                        small = (small + least) // 2
                P.sk_set_workspace(S.handle, ws.data_ptr(), least)
            Y = torch.full((k, 100), float("nan"), dtype=torch.float32, device="cuda")
            P.sk_apply_left(S.handle, Ad, m, n, 100, Y, 100)
            assert S.status() == 0
            assert rel_frob(Y[:, :n].cpu().numpy(), ref) <= TOL
            assert torch.isnan(Y[:, n:]).all()
        P.sk_set_workspace(S.handle, None, 0)
