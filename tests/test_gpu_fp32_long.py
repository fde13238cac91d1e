"""FP32 left sketch of a matrix of so many rows, and with so many tiles of Y, that
one accumulation runs over all of them.

Tolerance: a chain of the main sums is at most 16 truncated sums, below 2^-23
each of a running sum that is on average half the final one (1e-6 if all
pointed the same way); the cross sums, below 3 x 2^-9 of the whole, are at most
1280 such sums between two readings (5e-7); 4096 chains are added with IEEE
adds, each off by at most 2^-24 of the running sum, in either direction
(sqrt(4096) x 2^-24 x 0.58 = 2.2e-6)."""
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

TOL = 4e-6


@pytest.mark.parametrize("dist", [0, 1])
def test_error_does_not_grow_with_the_rows_of_a_split(dist):
    require_gpu()
    import paper_2603_20966_gb300 as P
    m, n, k, rows = 1 << 20, 64, 304 * 128, 64  # two tiles of Y per SM
    A = torch.randn((m, n), device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    with P.Sketch(3, dist, k, P.SK_FP32) as S:
        Y = S.left(A)
        assert S.status() == 0
        ref = torch.zeros((rows, n), dtype=torch.float64, device="cuda")
        for r0 in range(0, m, 1 << 16):
            ref += (S.materialize(0, r0, rows, 1 << 16).double() @
                    A[r0:r0 + (1 << 16)].double())
        ref *= S.scale
    assert rel_frob(Y[:rows].cpu().numpy(), ref.cpu().numpy()) <= TOL
