"""FP32 left sketch on the tensor cores (three BF16 values per FP32 operand)
against the FP64 oracle, at the edges of its tiles: rows of S (128 per tile),
columns (chunks of 64, at most 4 per tile), stages of 32 rows of m, chains of
at most 32 stages, more items than SMs; unaligned rows; special values.

Tolerance: both operands are exact, the products left out are below 3 x 2^-25
of the kept ones, and a chain adds at most 64 tensor-core sums, each truncated
by at most 2^-23 of a running sum that is on average half the final one: below
64 x 2^-24 = 3.8e-6 if every truncation pointed the same way."""
import numpy as np
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

G, R, U = 0, 1, 2
TOL = 4e-6


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


def _A(m, n, seed):
    from paper_2603_20966_gb300.workloads import gaussian_matrix
    return gaussian_matrix(m, n, seed, device="cpu")


def _left(P, seed, dist, k, A_cpu, lda=None, shift=0):
    m, n = A_cpu.shape
    lda = lda or n
    buf = torch.full((m * lda + shift,), float("nan"), dtype=torch.float32, device="cuda")
    A = buf[shift:].view(m, lda)
    A[:, :n] = A_cpu.cuda()
    Y = torch.full((k, n), float("nan"), dtype=torch.float32, device="cuda")
    with P.Sketch(seed, dist, k, P.SK_FP32) as S:
        P.sk_apply_left(S.handle, A, m, n, lda, Y, n)
        assert S.status() == 0
    return Y.cpu().numpy()


@pytest.mark.parametrize("dist", [G, R, U])
@pytest.mark.parametrize("k,m,n,lda,shift", [
    (128, 2048, 256, 256, 0), (129, 2049, 257, 258, 0), (127, 2047, 255, 257, 1),
    (64, 31, 64, 64, 0), (65, 33, 65, 65, 1), (256, 1024, 128, 128, 2), (300, 1056, 129, 131, 3),
    (666, 5003, 333, 333, 0), (32, 40001, 32, 32, 0), (1000, 6000, 700, 701, 0)])
def test_matches_oracle(P, orc, dist, k, m, n, lda, shift):
    A = _A(m, n, k + m + n)
    got = _left(P, 7, dist, k, A, lda, shift)
    assert rel_frob(got, orc.apply_left(7, dist, 0, k, A.numpy())) <= TOL


@pytest.mark.parametrize("scale", [2.0**-120, 2.0**-100, 2.0**100])
def test_magnitudes(P, orc, scale):
    # 2^-120: below what three BF16 values hold, multiplied in FP32 FMAs
    A = _A(1500, 80, 3)
    ref = orc.apply_left(7, G, 0, 70, A.numpy())
    got = _left(P, 7, G, 70, A * scale).astype(np.float64) / scale
    assert rel_frob(got, ref) <= TOL


def test_largest_and_special_values(P, orc):
    m, n, k = 600, 70, 40
    A = _A(m, n, 4)
    ref = orc.apply_left(7, G, 0, k, A.numpy())
    S = orc.generate(7, G, 0, 0, 0, k, m)
    A[17, 5], A[18, 6], A[19, 7] = float("inf"), float("-inf"), float("nan")
    A[20, 8], A[400, 8] = float("inf"), float("-inf")
    got = _left(P, 7, G, k, A)
    np.testing.assert_array_equal(got[:, 5], np.sign(S[:, 17]) * np.inf)
    np.testing.assert_array_equal(got[:, 6], -np.sign(S[:, 18]) * np.inf)
    assert np.isnan(got[:, 7]).all()
    opposite = np.sign(S[:, 20]) == np.sign(S[:, 400])
    assert np.isnan(got[opposite, 8]).all() and np.isinf(got[~opposite, 8]).all()
    keep = [j for j in range(n) if j not in (5, 6, 7, 8)]
    assert rel_frob(got[:, keep], ref[:, keep]) <= TOL
    # the largest finite values: no BF16 value is as large
    A = torch.zeros((m, n))
    A[3, :] = torch.finfo(torch.float32).max
    got = _left(P, 7, G, k, A)
    small = np.abs(S[:, 3]) < 0.99
    want = (S[small, 3].astype(np.float64) * float(A[3, 0]) * orc.scale(k))
    assert rel_frob(got[small], np.repeat(want[:, None], n, axis=1)) <= TOL


# (k, m, n): whose CUDA-core form needs more, or (one split) no workspace
@pytest.mark.parametrize("k,m,n", [(100, 9000, 90), (20, 200, 40)])
def test_lent_workspaces(P, orc, k, m, n):
    A = _A(m, n, 6)
    ref = orc.apply_left(7, G, 0, k, A.numpy())
    Ad = A.cuda()
    with P.Sketch(7, G, k, P.SK_FP32) as S:
        size = P.sk_workspace_size(S.handle, 0, m, n)
        ws = torch.empty(size + 64, dtype=torch.uint8, device="cuda")
        for lent in (size, 64 if (k, m, n) == (20, 200, 40) else size + 64):
            Y = torch.full((k, n), float("nan"), dtype=torch.float32, device="cuda")
            P.sk_set_workspace(S.handle, ws.data_ptr(), lent)
            P.sk_apply_left(S.handle, Ad, m, n, n, Y, n)
            assert S.status() == 0
            assert rel_frob(Y.cpu().numpy(), ref) <= TOL
        P.sk_set_workspace(S.handle, None, 0)


def test_same_bits_served_and_without_allocation(P):
    k, m, n = 70, 3001, 52
    A = _A(m, n, 8).cuda()
    with P.Sketch(7, G, k, P.SK_FP32) as S, P.Server(1 << 28) as server:
        Y, Z = S.left(A), torch.empty((k, n), dtype=torch.float32, device="cuda")
        P._native.sk_apply_left_noalloc(S.handle, A, m, n, n, Z, n)
        W = server.result(server.submit(S, A))
        assert S.status() == 0
        assert torch.equal(Y, Z) and torch.equal(Y, W)
