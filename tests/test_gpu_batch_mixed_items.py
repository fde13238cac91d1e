"""GPU parity of batches whose CTA pairs run many short items of alternating
distributions: Rademacher items (A split by the workers) behind Gaussian and
uniform ones (A split by the epilogue warps) on the ring with separate S
tiles, where a worker group that starts a Rademacher stage has not waited for
the A tiles before it."""
import random

import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

BF16 = 1
TOL = 1e-5


def _problems():
    """120 problems of all distributions, k <= 1024 (Gaussian and uniform
    ones split A in the kernel), with widths and lengths that put short items
    of every distribution next to each other in the list, longest first."""
    rng = random.Random(2024)
    probs = []
    for i in range(120):
        n = rng.choice([32, 63, 100, 256, 300, 512])
        probs.append((rng.randint(200, 1600), n, rng.choice([64, 200, 256, 300]), i % 3, 500 + i))
    probs[0] = (1200, 512, 1024, 0, 500)
    probs[1] = (1200, 512, 1024, 1, 501)
    return probs


@pytest.mark.parametrize("item_stages", [4, 8, 24])
def test_short_items_of_mixed_distributions(orc, item_stages):
    require_gpu()
    import paper_2603_20966_gb300 as P
    gen = torch.Generator(device="cuda").manual_seed(31)
    data = []
    b = P.sk_batch_create()
    for m, n, k, dist, seed in _problems():
        ld = (n + 3) // 4 * 4
        A = torch.randn((m, ld), device="cuda", generator=gen)
        Y = torch.full((k, ld), float("nan"), device="cuda")
        h = P.sk_create(seed, dist, k)
        P.sk_set_precision(h, BF16)
        P.sk_batch_add(b, h, A, m, n, ld, Y, ld)
        data.append((h, A, Y, m, n, k, dist, seed))
    P.sk_batch_set_config(b, item_stages, 512, 4)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    try:
        first = None
        for _ in range(20):
            for d in data:
                d[2].fill_(float("nan"))
            torch.cuda.synchronize()
            P.sk_batch_run(b, st)
            assert P.sk_batch_status(b, st) == 0
            ys = [Y[:, :n].clone() for _, _, Y, _, n, _, _, _ in data]
            if first is None:
                first = ys
            for y, f, d in zip(ys, first, data):
                assert torch.equal(y, f), d[3:]
        for y, (_, A, _, m, n, k, dist, seed) in zip(first, data):
            ref = orc.apply_left(seed, dist, BF16, k, A[:, :n].cpu().numpy())
            assert rel_frob(y.cpu().numpy(), ref) <= TOL, (m, n, k, dist)
    finally:
        P.sk_batch_destroy(b)
        for d in data:
            P.sk_destroy(d[0])
