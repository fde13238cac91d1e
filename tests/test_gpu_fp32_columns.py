"""FP32 left sketch of matrices whose columns differ in magnitude: each column
of Y to the form's own accuracy, whatever the columns beside it hold.  BF16
parts of elements below 2^-110 are subnormal, so a column that is small all
through an item has to be multiplied another way than a normal one.

Tolerance: that of test_gpu_fp32_tc, for each column by itself.  A column of
subnormal elements has sums on the grid of 2^-149, and a chain of FMAs rounds to it
once per row: m x 2^-150."""
import numpy as np
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

G, R, U = 0, 1, 2
TOL = 4e-6
SCALES = [1.0, 2.0**-120, 2.0**-112, 2.0**60, 2.0**-126, 2.0**-104, 2.0**-118]


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


def _check(P, orc, seed, dist, k, A, atol=None):
    m, n = A.shape
    with P.Sketch(seed, dist, k, P.SK_FP32) as S:
        Y = torch.full((k, n), float("nan"), dtype=torch.float32, device="cuda")
        S.left(A.cuda(), out=Y)
        assert S.status() == 0
    got = Y.cpu().numpy()
    ref = orc.apply_left(seed, dist, 0, k, A.numpy())
    for j in range(n):
        if atol is not None and np.abs(A[:, j].numpy()).max() < 2.0**-122:
            assert np.abs(got[:, j] - ref[:, j]).max() <= atol, j
        else:
            assert rel_frob(got[:, j], ref[:, j]) <= TOL, j


def _A(m, n, seed):
    return torch.randn((m, n), generator=torch.Generator().manual_seed(seed))


# one and several tiles of columns, one and several splits of m, more items
# than SMs
@pytest.mark.parametrize("dist", [G, R, U])
@pytest.mark.parametrize("k,m,n", [(70, 1500, 80), (130, 5003, 333), (64, 20000, 16),
                                   (3000, 300, 701), (20, 64, 7)])
def test_columns_of_different_magnitude(P, orc, dist, k, m, n):
    A = _A(m, n, k + m + n)
    for j in range(n):
        A[:, j] *= SCALES[j % len(SCALES)]
    _check(P, orc, 11, dist, k, A, atol=m * 2.0**-150)


def test_column_small_in_some_rows(P, orc):
    """Small in whole splits, in single rows, zero elsewhere, or beside zeros."""
    m, n = 8000, 72
    A = _A(m, n, 3)
    A[:4000, 3] *= 2.0**-120
    A[4000:, 5] *= 2.0**-120
    A[::2, 7] *= 2.0**-120
    A[:, 9] = 0.0
    A[77, 9] = 2.0**-117 * 1.2345678
    A[:, 11] *= 2.0**-120
    A[6000, 11] = float("nan")
    A[:, 13] *= 2.0**-120
    A[6000, 13] = 1.0
    k = 40
    with P.Sketch(5, G, k, P.SK_FP32) as S:
        Y = S.left(A.cuda()).cpu().numpy()
        assert S.status() == 0
    assert np.isnan(Y[:, 11]).all()
    A[:, 11] = 0.0
    Y[:, 11] = 0.0
    ref = orc.apply_left(5, G, 0, k, A.numpy())
    for j in range(n):
        assert rel_frob(Y[:, j], ref[:, j]) <= TOL, j


@pytest.mark.parametrize("exponent", [-110, -125, -135])
def test_whole_matrix_small(P, orc, exponent):
    m, n = 3000, 130
    A = (_A(m, n, 4).double() * 2.0**exponent).float()
    if exponent < -120:  # sums on the subnormal grid
        with P.Sketch(5, G, 64, P.SK_FP32) as S:
            Y = S.left(A.cuda()).cpu().numpy()
            assert S.status() == 0
        ref = orc.apply_left(5, G, 0, 64, A.numpy())
        assert np.abs(Y - ref).max() <= m * 2.0**-150
    else:
        _check(P, orc, 5, G, 64, A)


def test_small_matrix_of_many_rows_keeps_the_wait_limit(P):
    """A sketch of small elements takes no step that outlasts a (shortened)
    wait limit of the kernel."""
    m, n, k = 60000, 256, 152 * 128  # one item per SM
    A = (_A(m, n, 9).double() * 2.0**-115).float().cuda()
    with P.Sketch(5, G, k, P.SK_FP32) as S:
        P.sk_debug_set_wait(S.handle, 20_000_000, -1)
        Y = S.left(A)
        assert S.status() == 0
        ref = S.materialize(0, 0, 128, m).double() @ (A.double() * 2.0**115) * S.scale
    assert rel_frob(Y[:128].double().cpu().numpy() * 2.0**115, ref.cpu().numpy()) <= TOL
