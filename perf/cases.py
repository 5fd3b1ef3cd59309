"""The calls this library is measured on.

Each case is one pass through the public binding as an eigensolver makes it:
Gram products, the projection against a basis, CholQR and SVQB of a block, the
iterated two-phase algorithm, a batch of blocks, a burst of server requests.
Sizes, condition numbers and column counts are those of the benchmark's
workloads and of the tests (bench.py, synth.py); ``draw`` spreads them over the
same ranges.  Inputs are seeded on the GPU: a basis V with orthonormal columns,
blocks X = G diag(sigma) W^T with G a Gaussian / sqrt(n), W a Haar rotation and
sigma log-spaced from 1 to 1/kappa (condition number kappa up to a few percent).

In-place calls work on a copy that is made anew on every pass, as a solver's
block is new in every iteration.  Factors (R, Z) of a block are returned in FP64
(their high parts), as an FP64 solver takes them; Gram matrices and C = V^T Y as
the double-double pairs that the calls return.
"""
import math
import random

import torch

import paper_1806_01036_gb300 as eo

PREC = {"dd": eo.DD, "fp64": eo.FP64, "f32": eo.F32}


def listed():
    return [
        # the smallest call: one L2-resident block per iteration of a small eigenproblem (latency, launches, k x k step)
        {"name": "block_cholqr_100000x8", "op": "cholqr", "n": 100_000, "k": 8, "kappa": 1e6, "prec": "dd"},
        # the solver step of a large run: projection against 64 locked vectors, Gram and two-pass CholQR of a hard block
        {"name": "step_4000000x64x16", "op": "step", "n": 4_000_000, "kv": 64, "k": 16, "kappa": 1e10},
        # Gram matrix of a wide search space before a Rayleigh-Ritz step (the precision sweep's widest k)
        {"name": "gram_8000000x64", "op": "gram", "n": 8_000_000, "k": 64, "kappa": 1e8, "prec": "dd"},
        # Gram matrix of a few very long vectors (the sweep's narrow end)
        {"name": "gram_32000000x4", "op": "gram", "n": 32_000_000, "k": 4, "kappa": 1e8, "prec": "dd"},
        # projection of a packed block whose odd row count no 16-byte copy can address, ragged column counts
        {"name": "project_1500001x40x12", "op": "project", "n": 1_500_001, "kv": 40, "k": 12, "kappa": 1e4},
        # SVQB of one wide block: the eigensolve of a 32 x 32 Gram matrix between two streaming passes
        {"name": "svqb_1000000x32", "op": "svqb", "n": 1_000_000, "k": 32, "kappa": 1e6, "prec": "dd"},
        # the iterated two-phase algorithm on a runtime-figure shape (a basis of 20, blocks of 4)
        {"name": "iterate_4000000x20x4", "op": "iterate", "n": 4_000_000, "kv": 20, "k": 4, "kappa": 1e3, "kappa_xw": 1e6},
        # many independent blocks of uneven sizes in one graph launch
        {"name": "batch_svqb_48", "op": "batch", "blocks": 48, "nmin": 10_000, "nmax": 400_000, "kappa": 1e8},
        # a burst of requests to the server, each against its own resident basis
        {"name": "serve_burst_16", "op": "serve", "requests": 16, "nmin": 50_000, "nmax": 1_000_000, "kappa": 1e8},
        # B-inner product CholQR of a generalized problem's block, B X given
        {"name": "cholqr_b_1000000x16", "op": "cholqr_b", "n": 1_000_000, "k": 16, "kappa": 1e4},
        # plain FP64 CholQR2, for callers that keep to FP64 arithmetic
        {"name": "fp64_cholqr2_500000x16", "op": "cholqr", "n": 500_000, "k": 16, "kappa": 1e4, "prec": "fp64", "passes": 2},
        # FP32 blocks of the single-precision iterations
        {"name": "f32_cholqr_2000000x32", "op": "cholqr", "n": 2_000_000, "k": 32, "kappa": 1e2, "prec": "f32"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["cholqr", "step", "gram", "gram", "project", "svqb", "iterate", "batch", "serve", "cholqr_b", "fp64", "f32"])
    kappa = float("%.3g" % 10 ** rng.uniform(0.5, 10))
    if op == "cholqr":
        return {"op": "cholqr", "n": _logint(rng, 10_000, 4_000_000), "k": rng.randint(1, 32), "kappa": kappa, "prec": "dd"}
    if op == "step":
        kv = rng.randint(8, 64)
        return {"op": "step", "n": _logint(rng, 50_000, 4_000_000), "kv": kv, "k": rng.randint(2, max(2, kv // 4)), "kappa": kappa}
    if op == "gram":
        k = _logint(rng, 1, 64)
        return {"op": "gram", "n": _logint(rng, 100_000, min(32_000_000, 500_000_000 // k)), "k": k, "kappa": kappa, "prec": "dd"}
    if op == "project":
        return {"op": "project", "n": _logint(rng, 50_000, 2_000_000), "kv": rng.randint(4, 64), "k": rng.randint(1, 32), "kappa": min(kappa, 1e4)}
    if op == "svqb":
        return {"op": "svqb", "n": _logint(rng, 10_000, 2_000_000), "k": rng.randint(2, 32), "kappa": min(kappa, 1e6), "prec": "dd"}
    if op == "iterate":
        return {"op": "iterate", "n": _logint(rng, 100_000, 4_000_000), "kv": rng.randint(10, 40), "k": rng.randint(1, 4), "kappa": 1e3, "kappa_xw": 1e6}
    if op == "batch":
        return {"op": "batch", "blocks": rng.randint(8, 48), "nmin": 10_000, "nmax": _logint(rng, 50_000, 400_000), "kappa": kappa}
    if op == "serve":
        return {"op": "serve", "requests": rng.randint(2, 16), "nmin": 50_000, "nmax": _logint(rng, 100_000, 1_000_000), "kappa": kappa}
    if op == "cholqr_b":
        return {"op": "cholqr_b", "n": _logint(rng, 10_000, 1_000_000), "k": rng.randint(2, 32), "kappa": min(kappa, 1e4)}
    if op == "fp64":
        return {"op": "cholqr", "n": _logint(rng, 10_000, 1_000_000), "k": rng.randint(2, 24), "kappa": min(kappa, 1e4), "prec": "fp64", "passes": 2}
    return {"op": "cholqr", "n": _logint(rng, 10_000, 2_000_000), "k": rng.randint(8, 48), "kappa": min(kappa, 1e2), "prec": "f32"}


# ---------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _gauss(n, k, g):
    """Column-major n x k Gaussian of norm about 1 per column."""
    return (torch.randn((k, n), generator=g, device="cuda", dtype=torch.float64) / math.sqrt(n)).t()


def _basis(n, k, g):
    """n x k with orthonormal columns."""
    v = _gauss(n, k, g)
    for _ in range(2):
        w = torch.linalg.inv(torch.linalg.cholesky(v.t() @ v))
        v = (w @ v.t()).t()
    return v


def _block(n, k, kappa, g):
    """n x k block of condition number about kappa."""
    q, r = torch.linalg.qr(torch.randn((k, k), generator=g, device="cuda", dtype=torch.float64))
    sigma = torch.logspace(0, -math.log10(kappa), k, device="cuda", dtype=torch.float64)
    return ((q * sigma) @ _gauss(n, k, g).t()).t()


def _sizes(case):
    """Sizes of the members of a batch or a burst: rows log-uniform, columns as in the batched and serving workloads.
    They belong to the case; only the values come from the seed."""
    rng = random.Random(20180604)
    count = case["blocks"] if case["op"] == "batch" else case["requests"]
    ks = (4, 8, 16, 32) if case["op"] == "batch" else (8, 16, 32, 64)
    return [(_logint(rng, case["nmin"], case["nmax"]), rng.choice(ks)) for _ in range(count)]


def _inputs(case, seed):
    g = _gen(seed)
    op = case["op"]
    if op == "batch":
        return [_block(n, k, case["kappa"], g) for n, k in _sizes(case)]
    if op == "serve":
        return [(_basis(n, kv, g), _block(n, kv // 4, case["kappa"], g)) for n, kv in _sizes(case)]
    n, k = case["n"], case["k"]
    if op in ("step", "project"):
        return _basis(n, case["kv"], g), _block(n, k, case["kappa"], g)
    if op == "iterate":
        v = _basis(n, case["kv"], g)
        a = torch.randn((k, case["kv"]), generator=g, device="cuda", dtype=torch.float64)
        return v, (a @ v.t() + _block(n, k, case["kappa"], g).t() / case["kappa_xw"]).t()
    x = _block(n, k, case["kappa"], g)
    if op == "cholqr_b":  # B = tridiag(-0.2, 1, -0.2), applied by the caller
        bx = x.t().clone()
        bx[:, 1:] -= 0.2 * x.t()[:, :-1]
        bx[:, :-1] -= 0.2 * x.t()[:, 1:]
        return x, bx.t()
    if case.get("prec") == "f32":
        return x.t().float().contiguous().t()
    return x


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.ctx = case, eo.Context(0)
    s.inp = _inputs(case, seed)
    op = case["op"]
    if op == "batch":
        s.work = [x.t().clone().t() for x in s.inp]
        s.batch = eo.Batch(s.ctx, s.work, method=eo.BATCH_SVQB, passes=0, prec=eo.DD, tune=False)
    elif op == "serve":
        s.server = eo.Server(s.ctx, 100 << 30, slots=16)
        s.ids = [s.server.add_basis(v) for v, _ in s.inp]
        s.out = [torch.empty_like(y) for _, y in s.inp]
        s.r = [tuple(torch.zeros((y.shape[1],) * 2, dtype=torch.float64, device="cuda").t() for _ in range(2)) for _, y in s.inp]
        s.info = torch.zeros(len(s.inp), dtype=torch.int32, device="cuda")
    elif op in ("step", "project"):
        s.out = torch.empty_like(s.inp[1])
    elif op == "cholqr_b":
        s.work = tuple(x.t().clone().t() for x in s.inp)
    elif op == "iterate":
        s.work = s.inp[1].t().clone().t()
    elif op != "gram":
        s.work = s.inp.t().clone().t()
    torch.cuda.synchronize()
    return s


def run(s):
    c, op = s.case, s.case["op"]
    prec = PREC[c.get("prec", "dd")]
    if op == "gram":
        return eo.gram(s.ctx, s.inp, prec=prec)
    if op == "cholqr":
        s.work.copy_(s.inp)
        r, _, info = eo.cholqr(s.ctx, s.work, passes=c.get("passes", 0), prec=prec)
        return s.work, r, info
    if op == "svqb":
        s.work.copy_(s.inp)
        z, _, rank = eo.svqb(s.ctx, s.work, passes=0, prec=prec)
        return s.work, z, rank
    if op == "project":
        return eo.project(s.ctx, *s.inp, Yout=s.out)
    if op == "step":
        q, coef, m = eo.project(s.ctx, *s.inp, Yout=s.out)
        r, _, info = eo.cholqr(s.ctx, q, passes=0, M=m)
        return q, coef, m, r, info
    if op == "iterate":
        s.work.copy_(s.inp[1])
        iters, rank = eo.orthogonalize(s.ctx, s.inp[0], s.work)
        return s.work, iters, rank
    if op == "cholqr_b":
        s.work[0].copy_(s.inp[0])
        s.work[1].copy_(s.inp[1])
        r, _, info = eo.cholqr_b(s.ctx, *s.work, passes=0)
        return s.work[0], s.work[1], r, info
    if op == "batch":
        for w, x in zip(s.work, s.inp):
            w.copy_(x)
        s.batch.run()
        return s.work, s.batch.out
    ids = [s.server.submit(b, y, Yout=o, R=r, info=s.info[i : i + 1])
           for i, (b, (_, y), o, r) in enumerate(zip(s.ids, s.inp, s.out, s.r))]
    status = [s.server.wait(i)[0] for i in ids]
    return s.out, [r[0] for r in s.r], s.info, status


def work(case):
    op = case["op"]
    if op == "batch":
        return {"bytes": sum(16.0 * n * k for n, k in _sizes(case)), "flops": sum(4.0 * n * k * k for n, k in _sizes(case))}
    if op == "serve":
        return {"bytes": sum(8.0 * n * (kv + 2 * (kv // 4)) for n, kv in _sizes(case)),
                "flops": sum(4.0 * n * kv * (kv // 4) + 2.0 * n * (kv // 4) ** 2 for n, kv in _sizes(case))}
    n, k = float(case["n"]), case["k"]
    if op == "gram":
        return {"bytes": 8 * n * k, "flops": n * k * (k + 1)}
    if op in ("step", "project", "iterate"):
        kv = case["kv"]
        return {"bytes": 8 * n * (kv + 2 * k), "flops": 4 * n * kv * k + n * k * (k + 1) * (1 if op == "project" else 2)}
    width = 4 if case.get("prec") == "f32" else 8
    both = 2 if op == "cholqr_b" else 1
    return {"bytes": 2 * width * n * k * both, "flops": n * k * (k + 1) * (1 + both)}


# ------------------------------------------------- the same in plain torch


def _qr(x):
    q, r = torch.linalg.qr(x)
    s = torch.sign(torch.diagonal(r))
    return q * s, r * s[:, None]


def _polar(x):
    """(Q, Z) with Q = X Z the polar factor and Z = (X^T X)^{-1/2}."""
    q, r = torch.linalg.qr(x)
    u, s, wt = torch.linalg.svd(r)
    return q @ (u @ wt), (wt.t() / s) @ wt


def _project(v, y):
    c = v.t() @ y
    t = y - v @ c
    return t, c


def exact(case, seed):
    inp = _inputs(case, seed)
    op = case["op"]
    if op == "gram":
        return inp.t() @ inp, None
    if op == "cholqr":
        q, r = _qr(inp.double())
        return q, r, None
    if op == "svqb":
        q, z = _polar(inp)
        return q, z, None
    if op == "project":
        t, c = _project(*inp)
        return t, (c, None), (t.t() @ t, None)
    if op == "step":
        t, c = _project(*inp)
        q, r = _qr(t)
        return q, (c, None), (t.t() @ t, None), r, None
    if op == "iterate":
        return _polar(_project(inp[0], _project(*inp)[0])[0])[0], None, None
    if op == "cholqr_b":
        x, bx = inp
        m = x.t() @ bx
        w = torch.linalg.inv(torch.linalg.cholesky((m + m.t()) / 2))
        x1, bx1 = x @ w.t(), bx @ w.t()
        m = x1.t() @ bx1
        l2 = torch.linalg.cholesky((m + m.t()) / 2)
        w2 = torch.linalg.inv(l2)
        return x1 @ w2.t(), bx1 @ w2.t(), l2.t() @ torch.linalg.inv(w).t(), None
    if op == "batch":
        return [_polar(x)[0] for x in inp], None
    q = [_qr(_project(v, y)[0]) for v, y in inp]
    return [a for a, _ in q], [r for _, r in q], None, [None] * len(q)
