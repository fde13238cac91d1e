"""FP32 left sketches whose CUDA-core form needs no scratch (one split) where
handle-owned scratch cannot grow to what the tensor-core form takes: the first
call of a handle inside a stream capture, and a device without the memory.
Both are taken, as they are with a lent buffer that holds no more, and later
calls use the larger scratch again."""
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the FP32 form's


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


def _reference(S, A, rows):
    """Rows 0 .. rows - 1 of the sketch in 64 bits."""
    return (S.materialize(0, 0, rows, A.shape[0]).double() @ A.double() * S.scale).cpu().numpy()


def test_first_call_inside_a_capture(P):
    m, n, k = 100, 2000, 3000
    A = torch.randn(m, n, device="cuda")
    Y = torch.full((k, n), float("nan"), device="cuda")
    with P.Sketch(3, 0, k, P.SK_FP32) as S:
        ref = _reference(S, A, k)
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            S.left(A, out=Y)
        g.replay()
        torch.cuda.synchronize()
        assert S.status() == 0
        assert rel_frob(Y.cpu().numpy(), ref) <= TOL
        after = S.left(A)  # (scratch grows here)
        assert S.status() == 0
        assert rel_frob(after.cpu().numpy(), ref) <= TOL
        Y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert rel_frob(Y.cpu().numpy(), ref) <= TOL


def test_device_without_memory_for_the_partials(P):
    m, n, k = 64, 20000, 16384  # partials of 1.3 GB
    A = torch.randn(m, n, device="cuda")
    Y = torch.full((k, n), float("nan"), device="cuda")
    with P.Sketch(3, 0, k, P.SK_FP32) as S:
        ref = _reference(S, A, 128)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - (900 << 20), dtype=torch.uint8, device="cuda")
        try:
            S.left(A, out=Y)
            assert S.status() == 0
        finally:
            del hold
            torch.cuda.empty_cache()
        assert rel_frob(Y[:128].cpu().numpy(), ref) <= TOL
        Y.fill_(float("nan"))
        S.left(A, out=Y)
        assert S.status() == 0
        assert rel_frob(Y[:128].cpu().numpy(), ref) <= TOL
