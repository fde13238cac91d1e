"""Single sketches inside a caller's CUDA graph: their launches may begin while
the kernel before them is still running, which has to hold under capture too,
after a copy, a memset or another kernel, and on replay with new contents of
the same buffers."""
import pytest
import torch

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

G, R = 0, 1


@pytest.fixture(scope="module")
def P():
    require_gpu()
    import paper_2603_20966_gb300 as P
    return P


# one CTA per item; one pair per item; more items than pairs; right sketches
@pytest.mark.parametrize("side,form,dist,k,m,n", [
    ("left", 0, G, 64, 3000, 100), ("left", 1, G, 64, 4096, 256), ("left", 1, R, 100, 900, 300),
    ("left", 1, G, 300, 5000, 200), ("left", 1, R, 3000, 2000, 520), ("right", 0, G, 40, 600, 300),
    ("right", 1, G, 100, 2100, 500), ("right", 2, G, 64, 1100, 700)])
def test_capture_and_replay(P, side, form, dist, k, m, n):
    src = [torch.randn(m, n, device="cuda") for _ in range(2)]
    A = torch.empty(m, n, device="cuda")
    with P.Sketch(3, dist, k, form) as sk:
        go = sk.left if side == "left" else sk.right
        Y = torch.empty((k, n) if side == "left" else (m, k), device="cuda")
        want = [go(a).clone() for a in src]
        A.copy_(src[0])
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            Y.zero_()
            go(A, out=Y)        # after a memset or fill
            A.mul_(1.0)
            go(A, out=Y)        # after a kernel
            go(A, out=Y)        # after itself
        for a, w in zip(src, want):
            A.copy_(a)
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(Y, w)
        assert sk.status() == 0
