"""Overlapped launches in a caller's graph, with other data for every call: a
sketch that reads A before the kernel that writes it has finished, a reduction
that reads partials before its sketch has, or a sketch that overwrites the
partials of the call before it, gives another result than the same calls
waited for one by one."""
import pytest
import torch

from gpu_util import require_gpu

pytestmark = pytest.mark.gpu

G, R, U = 0, 1, 2


# large A (the copies take longer than a launch), one CTA per item, pairs with
# and without a work queue, few and many segments, quantized A
@pytest.mark.parametrize("side,form,dist,k,m,n", [
    ("left", 0, G, 64, 60000, 256), ("left", 0, R, 300, 5000, 333), ("left", 0, U, 16, 50, 20),
    ("left", 1, G, 64, 60000, 256), ("left", 1, U, 300, 20000, 300), ("left", 1, R, 3000, 9000, 520),
    ("right", 0, G, 40, 3000, 2000), ("right", 1, G, 100, 9000, 3000),
    ("right", 1, R, 100, 300, 5000), ("right", 2, G, 64, 9000, 3000)])
def test_every_call_of_a_graph_sees_its_own_data(side, form, dist, k, m, n):
    require_gpu()
    import paper_2603_20966_gb300 as P
    calls = 6
    gen = torch.Generator(device="cuda").manual_seed(5)
    src = [torch.randn(m, n, device="cuda", generator=gen) for _ in range(4)]
    A = torch.empty(m, n, device="cuda")
    ys = [torch.empty((k, n) if side == "left" else (m, k), device="cuda") for _ in range(calls)]
    with P.Sketch(3, dist, k, form) as sk:
        go = sk.left if side == "left" else sk.right
        want = []
        for a in src:
            A.copy_(a)
            torch.cuda.synchronize()
            want.append(go(A).clone())
            torch.cuda.synchronize()
        assert not torch.equal(want[0], want[1])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for i, y in enumerate(ys):
                if i % 3 == 2:                   # straight behind another sketch
                    go(src[i % 4], out=y)
                else:                            # behind the kernel that writes A
                    torch.mul(src[i % 4], 1.0, out=A)
                    go(A, out=y)
        for _ in range(5):
            A.fill_(float("nan"))
            for y in ys:
                y.fill_(float("nan"))
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            for i, y in enumerate(ys):
                assert torch.equal(y, want[i % 4]), i
        assert sk.status() == 0


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("side,form,k,m,n", [("left", 0, 64, 60000, 256), ("left", 1, 64, 60000, 256),
                                             ("right", 1, 100, 9000, 3000)])
def test_inputs_written_on_another_stream(side, form, k, m, n, captured):
    """A written on a second stream that the sketch's stream has waited for,
    and Y read there afterwards."""
    require_gpu()
    import paper_2603_20966_gb300 as P
    gen = torch.Generator(device="cuda").manual_seed(6)
    src = [torch.randn(m, n, device="cuda", generator=gen) for _ in range(3)]
    A = torch.empty(m, n, device="cuda")
    shape = (k, n) if side == "left" else (m, k)
    ys = [torch.empty(shape, device="cuda") for _ in src]
    copies = [torch.empty(shape, device="cuda") for _ in src]
    with P.Sketch(3, 0, k, form) as sk:
        go = sk.left if side == "left" else sk.right
        want = [go(a).clone() for a in src]
        torch.cuda.synchronize()
        other = torch.cuda.Stream()

        def steps():
            here = torch.cuda.current_stream()
            for a, y, c in zip(src, ys, copies):
                other.wait_stream(here)
                with torch.cuda.stream(other):
                    torch.mul(a, 1.0, out=A)
                here.wait_stream(other)
                go(A, out=y)
                other.wait_stream(here)
                with torch.cuda.stream(other):
                    c.copy_(y)
                here.wait_stream(other)
                go(src[0], out=y)

        for y in ys + copies:
            y.fill_(float("nan"))
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                steps()
            g.replay()
        else:
            steps()
        torch.cuda.synchronize()
        for y, c, w in zip(ys, copies, want):
            assert torch.equal(c, w)
            assert torch.equal(y, want[0])
        assert sk.status() == 0
