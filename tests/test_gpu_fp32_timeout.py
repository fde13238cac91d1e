"""Bounded waits of the FP32 left sketch on the tensor cores that run out: the
test-only hook sk_debug_set_wait shortens the limit and keeps one stage from
ever being handed to the MMA issuer.  The kernel gives up, records
SK_ETIMEOUT and the waiting site, waits for its own MMAs and copies in flight,
frees its tensor memory and exits; the next call on the handle is right."""
import time

import numpy as np
import pytest
import torch

from gpu_util import rel_frob, require_gpu

pytestmark = pytest.mark.gpu

LIMIT_NS = 20_000_000  # 20 ms: a healthy stage takes microseconds
TOL = 4e-6  # test_gpu_fp32_tc

# the MMA issuer waiting for the stage (0x22), a worker waiting for the slot it
# holds (0x43), an epilogue warp waiting for its chain (0x34)
SITES = {0x22, 0x43, 0x34}


# one item per block; several; the second run of an item with small elements
# (two stages in the first run)
@pytest.mark.parametrize("k,m,n,scale,stall", [
    (64, 4096, 96, 1.0, 1), (8000, 300, 701, 1.0, 4), (20, 64, 7, 2.0**-115, 0),
    (20, 64, 7, 2.0**-115, 2), (20, 64, 7, 2.0**-115, 3)])
def test_bounded_wait_gives_up_and_the_handle_recovers(orc, k, m, n, scale, stall):
    require_gpu()
    import paper_2603_20966_gb300 as P
    A_cpu = torch.randn((m, n), generator=torch.Generator().manual_seed(m)) * scale
    A = A_cpu.cuda()
    ref = orc.apply_left(7, 0, 0, k, A_cpu.numpy()) / scale
    with P.Sketch(7, 0, k, P.SK_FP32) as S:
        def check():
            Y = S.left(A)
            assert S.status() == 0
            assert rel_frob(Y.cpu().numpy().astype(np.float64) / scale, ref) <= TOL

        check()
        P.sk_debug_set_wait(S.handle, LIMIT_NS, stall)
        t0 = time.perf_counter()
        S.left(A)
        words = P.sk_debug_status(S.handle, torch.cuda.current_stream())
        assert time.perf_counter() - t0 < 5.0
        assert words[0] == 4, words  # SK_ETIMEOUT
        assert words[1] in SITES, hex(words[1])
        if words[1] == 0x22:
            assert words[2] == stall, words
        assert S.status() == 4  # reported once, then cleared
        P.sk_debug_set_wait(S.handle, 0, -1)
        for _ in range(2):
            check()
