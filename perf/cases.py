"""The work that users of this library have it do, as timed cases.

A case names an operation (left or right sketch, Nystrom pair, batch, request
server), an arithmetic form, a distribution and sizes.  Sizes are those of the
repository's own workloads (C1 to C5 and NYS of ``workloads.py``), and odd
ones of the same ranges.  ``exact`` restates the generator and the products
in torch, in 64 bits, sharing no code with the library.
"""
from __future__ import annotations

import math

import torch

import paper_2603_20966_gb300 as P

DISTS = {"gaussian": P.SK_GAUSSIAN, "rademacher": P.SK_RADEMACHER, "uniform": P.SK_UNIFORM}
FORMS = {"fp32": P.SK_FP32, "bf16": P.SK_BF16X2, "fp8": P.SK_FP8E4M3}
S_SEED = 7


def _case(op, form, dist, m, n, k, name=None):
    c = {"op": op, "form": form, "dist": dist, "m": m, "n": n, "k": k}
    return c if name is None else {"name": name, **c}


def _many(op, count, m_lo, m_hi, n_lo, n_hi, name=None):
    c = {"op": op, "form": "bf16", "count": count, "m_lo": m_lo, "m_hi": m_hi, "n_lo": n_lo,
         "n_hi": n_hi}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # one small sketch inside another program's step: launches and latency
        _case("left", "fp32", "gaussian", 4096, 256, 64, "left_small_fp32"),
        _case("left", "bf16", "gaussian", 4096, 256, 64, "left_small_bf16"),
        # an ordinary sketch at sizes that no tile divides, rows not 16-byte aligned
        _case("left", "fp32", "gaussian", 30011, 333, 666, "left_odd_fp32"),
        # the same in the tensor-core form: one member of C4 or C5 on its own
        _case("left", "bf16", "gaussian", 48611, 301, 602, "left_odd_bf16"),
        # compressing a very tall matrix (least squares, subspace embedding)
        _case("left", "bf16", "rademacher", 1 << 20, 512, 2048, "left_tall_rademacher"),
        _case("left", "bf16", "gaussian", 1 << 20, 512, 2048, "left_tall_gaussian"),
        # range finder of a large matrix of low numerical rank, near-FP32 and FP8
        _case("right", "bf16", "gaussian", 65536, 16384, 256, "right_range_finder"),
        _case("right", "fp8", "gaussian", 65536, 16384, 256, "right_range_finder_fp8"),
        # a smaller range finder with the uniform entries that the paper's runs draw
        _case("right", "bf16", "uniform", 20011, 3071, 100, "right_odd_uniform"),
        # the paper's Nystrom experiment: a kernel matrix of 50,000 points, r = 500
        _case("nystrom", "bf16", "gaussian", 50000, 50000, 500, "nystrom_kernel"),
        # many independent sketches of uneven shapes in one launch
        _many("batch", 256, 1024, 65536, 32, 512, "batch_uneven"),
        # a burst of requests at the server, results fetched
        _many("serve", 48, 1024, 1 << 18, 32, 512, "serve_burst"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["left", "left", "left", "right", "right", "nystrom", "batch", "serve"])
    dist = rng.choice(["gaussian", "gaussian", "rademacher", "uniform"])
    if op == "left":
        if rng.random() < 0.3:
            return _case("left", "fp32", dist, _log_int(rng, 1024, 65536), rng.randint(32, 512),
                         _log_int(rng, 64, 1024))
        return _case("left", "bf16", dist, _log_int(rng, 1024, 1 << 20), rng.randint(32, 512),
                     _log_int(rng, 64, 2048))
    if op == "right":
        form = rng.choice(["fp32", "bf16", "bf16", "fp8"])
        if form == "fp32":
            return _case("right", "fp32", dist, _log_int(rng, 1024, 16384),
                         _log_int(rng, 256, 4096), _log_int(rng, 16, 256))
        return _case("right", form, dist, _log_int(rng, 1024, 65536), _log_int(rng, 256, 16384),
                     _log_int(rng, 16, 256))
    if op == "nystrom":
        n = _log_int(rng, 2000, 50000)
        return _case("nystrom", "bf16", dist, n, n, _log_int(rng, 50, 500))
    if op == "batch":
        return _many("batch", _log_int(rng, 8, 256), 1024, _log_int(rng, 4096, 65536), 32,
                     rng.randint(96, 512))
    return _many("serve", _log_int(rng, 2, 48), 1024, _log_int(rng, 4096, 1 << 18), 32,
                 rng.randint(96, 512))


def _up4(x):
    return (x + 3) // 4 * 4


def _normal(m, n, ld, seed):
    """A[m x n] ~ N(0, 1) on the GPU in rows of ld elements."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty((m, ld), dtype=torch.float32, device="cuda").normal_(generator=g)[:, :n]


def _low_rank(m, n, ld, seed):
    """A = U V^T + 1e-3 E with rank 64 factors: what a range finder meets."""
    A = _normal(m, n, ld, seed).mul_(1e-3)
    U, V = _normal(m, 64, 64, seed + 1), _normal(n, 64, 64, seed + 2)
    for r0 in range(0, m, 8192):
        A[r0:r0 + 8192].addmm_(U[r0:r0 + 8192], V.t())
    return A


def _kernel_matrix(n, ld, seed):
    """RBF kernel matrix of n points ~ N(0, I_64), sigma = |X|_F / sqrt(n)."""
    X = _normal(n, 64, 64, seed)
    sq = (X * X).sum(dim=1)
    inv = -0.5 * n / sq.sum()
    K = torch.empty((n, ld), dtype=torch.float32, device="cuda")[:, :n]
    for r0 in range(0, n, 8192):
        blk = torch.mm(X[r0:r0 + 8192], X.t()).mul_(-2.0).add_(sq[r0:r0 + 8192, None]).add_(sq)
        K[r0:r0 + 8192] = blk.clamp_(min=0.0).mul_(inv).exp_()
    return K


def _problems(case):
    """(m, n, k, dist, seed) of a batch's or burst's members: m log-uniform,
    n uniform, k = 2n, a coin for the distribution.  A function of the case."""
    g = torch.Generator()
    g.manual_seed(1000)
    count = case["count"]
    u = torch.rand(count, generator=g, dtype=torch.float64)
    nn = torch.randint(case["n_lo"], case["n_hi"] + 1, (count,), generator=g)
    coin = torch.randint(0, 2, (count,), generator=g)
    lo, hi = math.log(case["m_lo"]), math.log(case["m_hi"])
    return [(int(round(math.exp(lo + float(u[i]) * (hi - lo)))), int(nn[i]), 2 * int(nn[i]),
             "rademacher" if coin[i] else "gaussian", 1000 + i) for i in range(count)]


def _input(case, seed):
    m, n = case["m"], case["n"]
    # the tensor-core forms take rows of whole 16-byte units
    ld = n if case["form"] == "fp32" else _up4(n)
    if case["op"] == "left":
        return _normal(m, n, ld, seed)
    return _kernel_matrix(n, ld, seed) if case["op"] == "nystrom" else _low_rank(m, n, ld, seed)


def _inputs(case, seed):
    return [_normal(m, n, _up4(n), seed * 1000 + i)
            for i, (m, n, _, _, _) in enumerate(_problems(case))]


class _State:
    pass


class _Batch:
    """A batch and its members' operators, released with the state."""

    def __init__(self):
        self.b = P.sk_batch_create()

    def __del__(self):
        P.sk_batch_destroy(self.b)


def prepare(case, seed):
    s = _State()
    s.op = case["op"]
    form = FORMS[case["form"]]
    if s.op in ("batch", "serve"):
        probs = _problems(case)
        s.A = _inputs(case, seed)
        s.sketches = [P.Sketch(sd, DISTS[d], k, form) for (_, _, k, d, sd) in probs]
        if s.op == "serve":
            s.server = P.Server(16 << 30)
            return s
        # every Y in one buffer, rows padded to 16-byte units
        sizes = [k * _up4(n) for (_, n, k, _, _) in probs]
        s.Y = torch.zeros(sum(sizes), dtype=torch.float32, device="cuda")
        s.batch, s.stream, at = _Batch(), torch.cuda.Stream(), 0
        for A, sk, (m, n, k, _, _), size in zip(s.A, s.sketches, probs, sizes):
            P.sk_batch_add(s.batch.b, sk.handle, A, m, n, A.stride(0), s.Y[at:], _up4(n))
            at += size
        return s
    s.A = _input(case, seed)
    s.sketch = P.Sketch(S_SEED, DISTS[case["dist"]], case["k"], form)
    s.out = None
    cols = case["n"] if s.op == "left" else case["k"]
    if s.op != "nystrom" and case["form"] != "fp32" and cols % 4:
        rows = case["k"] if s.op == "left" else case["m"]
        s.out = torch.empty((rows, _up4(cols)), dtype=torch.float32, device="cuda")[:, :cols]
    return s


def run(s):
    if s.op == "left":
        return s.sketch.left(s.A, out=s.out)
    if s.op == "right":
        return s.sketch.right(s.A, out=s.out)
    if s.op == "nystrom":
        return s.sketch.nystrom(s.A)
    if s.op == "batch":  # graphs are captured on a created stream
        here = torch.cuda.current_stream()
        s.stream.wait_stream(here)
        P.sk_batch_run(s.batch.b, s.stream)
        here.wait_stream(s.stream)
        return s.Y
    tickets = [s.server.submit(sk, A) for sk, A in zip(s.sketches, s.A)]
    return [s.server.result(t) for t in tickets]


def work(case):
    if case["op"] in ("batch", "serve"):
        p = _problems(case)
        return {"bytes": sum(4 * (m * n + k * n) for m, n, k, _, _ in p),
                "flops": sum(2 * k * m * n for m, n, k, _, _ in p)}
    m, n, k = case["m"], case["n"], case["k"]
    if case["op"] == "nystrom":
        return {"bytes": 4 * (n * n + n * k + k * k), "flops": 2 * n * n * k + 2 * n * k * k}
    y = k * n if case["op"] == "left" else m * k
    return {"bytes": 4 * (m * n + y), "flops": 2 * k * m * n}


# ---- the same results in 64 bits ----

_LOW = 0xFFFFFFFF


def _r32(x):
    """Rounded to FP32, kept in 64 bits."""
    return x.float().double()


def _fma(a, b, c):
    return _r32(a * b + c)


def _philox(seed, rows, j0, j1, dev):
    """Philox4x32-10 words of counters (j, r, 0, 0), each [rows, j1 - j0]."""
    c0 = torch.arange(j0, j1, dtype=torch.int64, device=dev)[None, :]
    c1 = torch.arange(rows, dtype=torch.int64, device=dev)[:, None]
    c2 = c3 = torch.zeros((1, 1), dtype=torch.int64, device=dev)
    k0, k1 = seed & _LOW, (seed >> 32) & _LOW
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _LOW) ^ c1 ^ k0, p1 & _LOW,
                          ((p0 >> 32) & _LOW) ^ c3 ^ k1, p0 & _LOW)
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return c0, c1, c2, c3


def _hex(text):
    return tuple(float.fromhex(v) for v in text.split())


_LN = _hex("-0x1.321a48p-4 0x1.068b28p-3 -0x1.0f9b0cp-3 0x1.22bf86p-3 -0x1.5424e0p-3 "
           "0x1.999fc2p-3 -0x1.000422p-2 0x1.555558p-2 -0x1.fffff8p-2")
_LN2_HI, _LN2_LO = _hex("0x1.62e4p-1 0x1.7f7d1cp-20")
_SIN = _hex("0x1.507834p-4 -0x1.32d2ccp-1 0x1.466bc6p+1 -0x1.4abbcep+2 0x1.921fb6p+1")
_COS = _hex("-0x1.a6d1f2p-6 0x1.e1f506p-3 -0x1.55d3c8p+0 0x1.03c1f0p+2 -0x1.3bd3ccp+2 0x1p+0")


def _horner(x, coeffs):
    p = torch.full_like(x, coeffs[0])
    for c in coeffs[1:]:
        p = _fma(x, p, c)
    return p


def _box_muller(xa, xb):
    """The two Gaussian entries of a pair of words, each FP32 step rounded."""
    u1 = (((xa >> 8) + 1).double() * 2.0**-24).float()
    i = u1.view(torch.int32).long() + 0x4AFB0C
    e = ((i >> 23) - 127).double()
    t = ((i & 0x7FFFFF) + 0x3F3504F4).int().view(torch.float32).double() - 1.0
    lnf = _fma(_r32(t * t), _horner(t, _LN), t)
    ln = _fma(e, _LN2_HI, _fma(e, _LN2_LO, lnf))
    rho = _r32(torch.sqrt(-2.0 * ln))
    r = ((xb >> 8) & 0x3FFFFF).double() * 2.0**-23 - 0.25
    r2 = _r32(r * r)
    sn, cs = _r32(r * _horner(r2, _SIN)), _horner(r2, _COS)
    turn = (xb >> 30) & 1 == 1
    rho = torch.where((xb >> 31) & 1 == 1, -rho, rho)
    return _r32(rho * torch.where(turn, -sn, cs)), _r32(rho * torch.where(turn, cs, sn))


def _entries(seed, dist, form, rows, c0, c1, dev):
    """g(r, c) for r < rows, c0 <= c < c1 (c0 a multiple of 128), in 64 bits,
    rounded to the stored precision of the form."""
    if dist == "rademacher":
        w = torch.stack(_philox(seed, rows, c0 // 128, (c1 + 127) // 128, dev), dim=-1)
        bits = (w[..., None] >> torch.arange(32, device=dev)) & 1
        return (1 - 2 * bits).reshape(rows, -1)[:, :c1 - c0].double()
    x = _philox(seed, rows, c0 // 4, (c1 + 3) // 4, dev)
    if dist == "uniform":
        g = torch.stack([(v >> 8).double() * 2.0**-24 for v in x], dim=-1)
    else:
        g = torch.stack(_box_muller(x[0], x[1]) + _box_muller(x[2], x[3]), dim=-1)
    g = g.reshape(rows, -1)[:, :c1 - c0].float()
    if form == "bf16":
        g = g.bfloat16().float()
    elif form == "fp8":
        g = g.to(torch.float8_e4m3fn).float()
    return g.double()


def _scale(k):
    one = torch.tensor(1.0, dtype=torch.float32)
    return float(one / torch.sqrt(torch.tensor(float(k), dtype=torch.float32)))


def _chunks(total, rows):
    step = max(128, (1 << 26) // rows // 128 * 128)
    return [(c, min(total, c + step)) for c in range(0, total, step)]


def _left(A, seed, dist, form, k):
    m, n = A.shape
    Y = torch.zeros((k, n), dtype=torch.float64, device=A.device)
    for c0, c1 in _chunks(m, k):
        Y.addmm_(_entries(seed, dist, form, k, c0, c1, A.device), A[c0:c1].double())
    return Y.mul_(_scale(k))


def _right(A, seed, dist, form, k):
    m, n = A.shape
    if form == "fp8":
        # one power-of-two scale per row: max |a| <= 448 * 2^e, then E4M3 codes
        e = torch.frexp(A.abs().amax(dim=1, keepdim=True).double() / 448.0)
        e = (e.exponent - (e.mantissa == 0.5).int()).double()
    Y = torch.zeros((m, k), dtype=torch.float64, device=A.device)
    for c0, c1 in _chunks(n, max(k, m)):
        a = A[:, c0:c1].double()
        if form == "fp8":
            a = (a * torch.exp2(-e)).float().to(torch.float8_e4m3fn).double()
        Y.addmm_(a, _entries(seed, dist, form, k, c0, c1, A.device).t())
    if form == "fp8":
        Y.mul_(torch.exp2(e))
    return Y.mul_(_scale(k))


def exact(case, seed):
    form = case["form"]
    if case["op"] in ("batch", "serve"):
        Y = [_left(A, sd, d, form, k)
             for A, (_, _, k, d, sd) in zip(_inputs(case, seed), _problems(case))]
        if case["op"] == "serve":
            return Y
        return torch.cat([torch.nn.functional.pad(y, (0, _up4(y.shape[1]) - y.shape[1])).reshape(-1)
                          for y in Y])
    A = _input(case, seed)
    if case["op"] == "left":
        return _left(A, S_SEED, case["dist"], form, case["k"])
    B = _right(A, S_SEED, case["dist"], form, case["k"])
    if case["op"] == "right":
        return B
    return B, _left(B, S_SEED, case["dist"], form, case["k"])
