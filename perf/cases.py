"""What a user of this library has it do, as timed cases: solves of ridge problems through the
Python binding (dense FP64, dense FP32 on the tensor cores, sparse CSR, batches of uneven
problems) and the Gram pass alone, over the sizes of the benchmark's configurations and tests.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed, ``run`` is
one call of the library and returns the vectors it computes, ``work`` counts what the call cannot
do without, ``exact`` gives the same results in 64-bit torch (one block update at a time, as
Algorithms 1 and 3 write them, with the sampler in numpy).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1612_04003_gb300 as ca

SEED = 42  # of the block sampler, as the benchmark sets it


def listed():
    return [
        # the smallest problem of the benchmark family, FP64: launch latency and short vectors;
        # the plain method (s = 1) and the s-step form of the same solve
        dict(name="tiny_f64_s1", kind="primal", dtype="f64", prec="f64", d=64, n=1024, cond=1.0,
             b=4, s=1, H=200, lam=1e-3, every=0, check=0, panels=False, warm=False),
        dict(name="tiny_f64_s4", kind="primal", dtype="f64", prec="f64", d=64, n=1024, cond=1.0,
             b=4, s=4, H=200, lam=1e-3, every=0, check=0, panels=False, warm=False),
        # the exact path on a problem of some size (the reference of a precision study), ragged,
        # with the recomputation of the residual vector every 8 outer steps
        dict(name="f64_ragged", kind="primal", dtype="f64", prec="f64", d=2003, n=24001, cond=1e4,
             b=16, s=8, H=128, lam=1e-6, every=8, check=0, panels=False, warm=False),
        # the same arithmetic in the dual method, more features than samples, from a warm start
        dict(name="f64_dual", kind="dual", dtype="f64", prec="f64", d=8190, n=1500, cond=1.0,
             b=8, s=4, H=256, lam=1e-2, every=0, check=0, panels=False, warm=True),
        # the headline: FP32 X in the library's panels, BF16x3 Gram, s = 16
        dict(name="headline_s16", kind="primal", dtype="f32", prec="bf16x3", d=4096, n=262144,
             cond=1e3, b=8, s=16, H=4096, lam=1e-4, every=0, check=0, panels=True, warm=False),
        # larger blocks on the same matrix, FP32-faithful split Gram
        dict(name="blocks32_s4", kind="primal", dtype="f32", prec="3xtf32", d=4096, n=262144,
             cond=1e3, b=32, s=4, H=256, lam=1e-4, every=0, check=0, panels=True, warm=False),
        # the precision study: row-major X (each call packs it), scaled FP16 Gram, s b = 256,
        # recomputation every 8 outer steps
        dict(name="precision_s16", kind="primal", dtype="f32", prec="fp16_scaled", d=8192,
             n=131072, cond=1e4, b=16, s=16, H=512, lam=1e-6, every=8, check=0, panels=False,
             warm=False),
        # a request of the served sizes solved alone: ragged, row-major, warm start, the stopping
        # test every 8 outer steps
        dict(name="served_dual", kind="dual", dtype="f32", prec="bf16x3", d=1000, n=20003,
             cond=1.0, b=8, s=16, H=1024, lam=1e-2, every=0, check=8, panels=False, warm=True),
        # the sparse dual (CSR of X^T, Pareto-distributed features) at two depths
        dict(name="sparse_s8", kind="csr", d=131072, n=16384, density=0.005, b=8, s=8, H=2048,
             lam=1e-5, every=0, check=0),
        dict(name="sparse_s32", kind="csr", d=131072, n=16384, density=0.005, b=8, s=32, H=2048,
             lam=1e-5, every=0, check=0),
        # a group of uneven requests in shared launches, as the serving loop groups them
        dict(name="batch_8", kind="batch", prec="bf16x3", count=8, sizes=5, d0=256, d1=2048,
             n0=4096, n1=32768, rows=64, Hmax=512),
        # the Gram and projection of one outer step alone, for programs with their own solver
        dict(name="gram_alone", kind="gram", dtype="f32", prec="tf32", d=1024, n=16384, rows=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds of call, sizes log-uniform over their ranges."""
    kind = rng.choice(["f64", "f64", "f32", "f32", "f32", "csr", "batch", "gram"])
    if kind == "f64":
        b = rng.choice([2, 4, 8, 16])
        s = rng.choice([v for v in (1, 4, 8, 16) if v * b <= 128])
        return dict(kind=rng.choice(["primal", "dual"]), dtype="f64", prec="f64",
                    d=_log(rng, 64, 2000), n=_log(rng, 512, 24000), cond=rng.choice([1.0, 1e2, 1e4]),
                    b=b, s=s, H=s * rng.randint(4, 50) + rng.randint(0, s - 1),
                    lam=10.0 ** rng.uniform(-4, -1), every=rng.choice([0, 0, 8]),
                    check=rng.choice([0, 0, 8]), panels=False, warm=rng.random() < 0.3)
    if kind == "f32":
        kind, panels = rng.choice(["primal", "dual"]), rng.random() < 0.5
        d, n = _log(rng, 256, 8192), _log(rng, 4096, 131072)
        n = min(n, (1 << 29) // d)
        if kind == "dual" and not panels:
            d = d // 4 * 4  # row-major X^T: rows of 16 bytes
        b = rng.choice([4, 8, 16, 32])
        s = rng.choice([v for v in (1, 4, 8, 16, 32) if v * b <= 256])
        return dict(kind=kind, dtype="f32",
                    prec=rng.choice(["bf16x3", "bf16x3", "3xtf32", "tf32", "fp16_scaled"]),
                    d=d, n=n, cond=rng.choice([1.0, 1e2, 1e4]), b=b, s=s,
                    H=s * rng.randint(8, 64), lam=10.0 ** rng.uniform(-4, -1),
                    every=rng.choice([0, 0, 8]), check=rng.choice([0, 0, 8]),
                    panels=panels, warm=rng.random() < 0.3)
    if kind == "csr":
        s = rng.choice([1, 4, 8, 16, 32])
        return dict(kind="csr", d=_log(rng, 8192, 131072), n=_log(rng, 2048, 16384),
                    density=rng.choice([0.002, 0.005]), b=rng.choice([4, 8]), s=s,
                    H=s * rng.randint(8, 60), lam=10.0 ** rng.uniform(-5, -2),
                    every=rng.choice([0, 0, 8]), check=rng.choice([0, 0, 8]))
    if kind == "batch":
        return dict(kind="batch", prec=rng.choice(["bf16x3", "3xtf32"]), count=rng.randint(2, 12),
                    sizes=rng.randrange(1 << 20), d0=256, d1=2048, n0=4096, n1=32768,
                    rows=rng.choice([32, 64, 128]), Hmax=256)
    prec = rng.choice(["tf32", "bf16x3", "3xtf32", "f64"])
    n = _log(rng, 1000, 65536)
    return dict(kind="gram", dtype="f64" if prec == "f64" else "f32", prec=prec,
                d=_log(rng, 256, 4096), n=n if prec == "f64" else n // 4 * 4,
                rows=rng.choice([8, 32, 100, 128, 256]))


# ---------------------------------------------------------------- inputs
def _problems(case):
    """The problems of a batch: sizes, method, block size, lambda (plain values)."""
    r = random.Random(case["sizes"])
    out = []
    for i in range(case["count"]):
        d = _log(r, case["d0"], case["d1"]) // 4 * 4
        n = _log(r, case["n0"], case["n1"]) // 4 * 4
        b, kind = r.choice([4, 8, 16]), "primal" if i % 2 == 0 else "dual"
        N = d if kind == "primal" else n
        out.append(dict(kind=kind, dtype="f32", d=d, n=n, cond=1.0, b=b, s=case["rows"] // b,
                        H=min(case["Hmax"], 4 * N // b), lam=10.0 ** r.uniform(-4, -1),
                        every=0, check=0, panels=False, warm=False, prec=case["prec"]))
    return out


def _dense(case, g):
    """X in the orientation of the method (primal d x n, dual n x d), the labels and the start.
    Rows of X^T scaled geometrically to the condition number, y = X^T w_true + 1% noise."""
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    d, n, primal = case["d"], case["n"], case["kind"] == "primal"
    rows, cols = (d, n) if primal else (n, d)
    ld = cols if case["dtype"] == "f64" else (cols + 3) // 4 * 4  # FP32: rows of 16 bytes
    A = torch.randn(rows, ld, generator=g, device="cuda", dtype=dt)
    scale = torch.logspace(0, -math.log10(case["cond"]), d, device="cuda", dtype=torch.float64).to(dt)
    A.mul_(scale[:, None] if primal else torch.nn.functional.pad(scale, (0, ld - d))[None, :])
    w = torch.randn(d, generator=g, device="cuda", dtype=dt)
    y = (w @ A[:, :n] if primal else A[:, :d] @ w).double()
    y += 0.01 * y.square().mean().sqrt() * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    x0 = torch.zeros(rows, device="cuda", dtype=torch.float64)
    if case["warm"]:
        x0 += 0.1 * torch.randn(rows, generator=g, device="cuda", dtype=torch.float64)
    return A, y, x0, cols


def _sparse(case, g):
    """CSR of X^T: feature f is in about min(n, k/U) samples (a Pareto tail), values N(0,1)."""
    d, n = case["d"], case["n"]
    ks = np.arange(1, n, dtype=np.float64)
    lo, hi = 1e-9, float(n)
    for _ in range(60):  # mean of the feature counts = density * n
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 1.0 + np.minimum(1.0, mid / ks).sum() < case["density"] * n else (lo, mid)
    u = 1.0 - torch.rand(d, generator=g, device="cuda", dtype=torch.float64)
    k = torch.clamp(torch.ceil(lo / u), max=n).long()
    heavy = k > n // 8
    f = torch.nonzero(heavy).flatten()
    m = torch.rand(f.numel(), n, generator=g, device="cuda") < (k[f] / n).float()[:, None]
    hf, hp = torch.nonzero(m, as_tuple=True)
    lf = torch.repeat_interleave(torch.arange(d, device="cuda"), torch.where(heavy, 0, k))
    lp = torch.randint(0, n, (lf.numel(),), generator=g, device="cuda")
    key = torch.unique(torch.cat([hp * d + f[hf], lp * d + lf]))  # by sample, then feature
    row, col = key // d, (key % d).int()
    val = torch.randn(key.numel(), generator=g, device="cuda", dtype=torch.float32)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    y = torch.randint(0, 2, (n,), generator=g, device="cuda").double() * 2 - 1
    return rowptr, col, val, row, y


def _gram_inputs(case, g):
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    A = torch.randn(case["d"], case["n"], generator=g, device="cuda", dtype=dt)
    idx = torch.randperm(case["d"], generator=g, device="cuda")[:case["rows"]].int()
    v = torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
    return A, idx, v


class _State:
    """A context on a stream of its own, as a program that solves repeatedly keeps it."""

    def __init__(self, case):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.ctx = ca.Context(0, stream=self.stream.cuda_stream)


def _vec(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    """The inputs on the GPU, the result vectors and the context that keeps its scratch."""
    st = _State(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "csr":
        rowptr, col, val, _, st.y = _sparse(case, g)
        st.X = (rowptr, col, val)
        st.x, st.aux = _vec(case["n"]), _vec(case["d"])
    elif case["kind"] == "gram":
        st.A, st.idx, st.v = _gram_inputs(case, g)
        r = st.idx.numel()
        st.G, st.p = torch.empty(r, r, dtype=torch.float64, device="cuda"), _vec(r)
    elif case["kind"] == "batch":
        st.problems = []
        for p in _problems(case):
            A, y, x0, cols = _dense(p, g)
            used = {"n": cols} if p["kind"] == "primal" else {"d": cols}
            st.problems.append(dict(method=p["kind"], X=A, y=y, x=_vec(A.shape[0]), aux=_vec(cols),
                                    b=p["b"], s=p["s"], H=p["H"], lam=p["lam"], seed=SEED,
                                    prec=p["prec"], **used))
    else:
        A, st.y, st.x0, cols = _dense(case, g)
        st.x, st.aux = _vec(A.shape[0]), _vec(cols)
        st.X = A
        st.kw = dict(b=case["b"], s=case["s"], H=case["H"], lam=case["lam"], seed=SEED,
                     prec=case["prec"], recompute_every=case["every"], check_every=case["check"])
        if case["panels"]:
            P = torch.empty((cols + 31) // 32 * A.shape[0] * 32, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            st.X = st.ctx.ca_pack_panels(A, P, K=cols)
            st.kw["panels"] = (A.shape[0], cols)
        elif case["kind"] == "primal":
            st.kw["n"] = cols
        torch.cuda.synchronize()  # A is read by the packing on the context's stream
    torch.cuda.synchronize()
    return st


def run(st):
    """One call of the library from the case's starting point; its output vectors."""
    case = st.case
    with torch.cuda.stream(st.stream):
        if case["kind"] == "gram":
            st.ctx.ca_gram_project(st.A, st.idx, st.v, st.G, st.p, prec=case["prec"])
            return {"G": st.G, "p": st.p}
        if case["kind"] == "batch":
            for p in st.problems:
                p["x"].zero_()
            st.ctx.ca_batch_solve(st.problems)
            return [{"x": p["x"], "aux": p["aux"]} for p in st.problems]
        if case["kind"] == "csr":
            st.x.zero_()
            st.ctx.ca_bdcd_solve(st.X, st.y, st.x, st.aux, b=case["b"], s=case["s"], H=case["H"],
                                 lam=case["lam"], seed=SEED, prec="f64", d=case["d"],
                                 recompute_every=case["every"], check_every=case["check"])
        else:
            st.x.copy_(st.x0)
            solve = st.ctx.ca_bcd_solve if case["kind"] == "primal" else st.ctx.ca_bdcd_solve
            solve(st.X, st.y, st.x, st.aux, **st.kw)
        return {"x": st.x, "aux": st.aux}


# ---------------------------------------------------------------- what a call cannot do without
def work(case):
    """Bytes: the sampled rows' values once (each row of X at most once, whatever the steps), the
    vectors in and out once.  Flops: per outer step the lower triangle of the Gram, the
    projection and the deferred update; for the sparse dual the projection and the update of
    every sampled entry and the products of the expected shared ones."""
    if case["kind"] == "batch":
        w = [work(p) for p in _problems(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    el = 8 if case.get("dtype") == "f64" else 4
    if case["kind"] == "gram":
        r, K = case["rows"], case["n"]
        return {"bytes": r * K * el + K * 8 + r * r * 8 + r * 8, "flops": r * (r + 1) * K + 2 * r * K}
    H, sb = case["H"], min(case["s"], case["H"]) * case["b"]
    if case["kind"] == "csr":
        per_row = case["density"] * case["d"]
        rows = min(case["n"], H * case["b"])
        return {"bytes": rows * per_row * 8 + 8 * (3 * case["n"] + case["d"]),
                "flops": H * case["b"] * (4 * per_row + 0.05 * per_row * sb)}
    N, K = (case["d"], case["n"]) if case["kind"] == "primal" else (case["n"], case["d"])
    passes = 1 + bool(case["warm"]) + case["kind"].count("primal")
    if case["every"]:
        passes += H // case["s"] // case["every"]
    if case["check"]:
        passes += 2 * (1 + H // case["s"] // case["check"])
    full = passes > 1  # the final X^T w, a recomputation or a check reads all of X
    rows = N if full else min(N, H * case["b"])
    return {"bytes": rows * K * el + 8 * (3 * N + 2 * K),
            "flops": H * case["b"] * K * (sb + 1 + 4) + 2 * (passes - 1) * N * K}


# ---------------------------------------------------------------- the same results in 64 bits
def _mulhi(a, b):
    m = np.uint64(0xFFFFFFFF)
    h = np.uint64(32)
    al, ah, bl, bh = a & m, a >> h, b & m, b >> h
    t = al * bl
    k = ah * bl + (t >> h)
    w = al * bh + (k & m)
    return ah * bh + (k >> h) + (w >> h)


def _philox(h, m4):
    """Philox4x64-10 words at counters (h, m4, 0, 0), key (SEED, 0)."""
    A, B = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    k0, k1 = SEED, 0
    x = [h, np.full_like(h, m4), np.zeros_like(h), np.zeros_like(h)]
    for _ in range(10):
        pa, pb = x[0], x[2]
        x = [_mulhi(B, pb) ^ x[1] ^ np.uint64(k0), B * pb, _mulhi(A, pa) ^ x[3] ^ np.uint64(k1), A * pa]
        k0 = (k0 + 0x9E3779B97F4A7C15) % 2**64
        k1 = (k1 + 0xBB67AE8584CAA73B) % 2**64
    return x


def _blocks(H, b, N):
    """H blocks of b distinct indices of [0, N): Floyd's algorithm on the Philox words."""
    h = np.arange(H, dtype=np.uint64)
    out = np.empty((H, b), dtype=np.int64)
    for m in range(b):
        if m % 4 == 0:
            words = _philox(h, m // 4)
        J = N - b + m
        t = _mulhi(words[m % 4], np.uint64(J + 1)).astype(np.int64)
        out[:, m] = np.where((out[:, :m] == t[:, None]).any(1), J, t)
    return torch.from_numpy(out).cuda()


def _exact_dense(case, A, y, x0, cols):
    """Algorithm 1 (primal) / Algorithm 3 (dual), one block at a time, FP64."""
    A = A[:, :cols]
    x = x0.clone()
    N, lam, b = A.shape[0], case["lam"], case["b"]
    step = max(1, (1 << 27) // cols)

    def xt(u):  # A^T u
        v = torch.zeros(cols, dtype=torch.float64, device="cuda")
        for r in range(0, N, step):
            v += u[r:r + step] @ A[r:r + step].double()
        return v

    blocks = _blocks(case["H"], b, N)
    eye = torch.eye(b, dtype=torch.float64, device="cuda")
    if case["kind"] == "primal":
        n = case["n"]
        rho = y - xt(x)
        for I in blocks:
            Y = A[I].double()
            dl = torch.linalg.solve(Y @ Y.T / n + lam * eye, Y @ rho / n - lam * x[I])
            x[I] += dl
            rho -= dl @ Y
        return {"x": x, "aux": xt(x)}
    c = 1.0 / (lam * case["n"])
    w = -c * xt(x)
    for I in blocks:
        Y = A[I].double()
        dl = torch.linalg.solve(c * (Y @ Y.T) + eye, Y @ w - x[I] - y[I])
        x[I] += dl
        w -= c * (dl @ Y)
    return {"x": x, "aux": w}


def exact(case, seed):
    """What ``run`` returns for these inputs, in 64-bit torch."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "gram":
        A, idx, v = _gram_inputs(case, g)
        Y = A[idx.long()].double()
        return {"G": Y @ Y.T, "p": Y @ v}
    if case["kind"] == "batch":
        out = []
        for p in _problems(case):
            out.append(_exact_dense(p, *_dense(p, g)))
        return out
    if case["kind"] == "csr":
        _, col, val, row, y = _sparse(case, g)
        A = torch.zeros(case["n"], case["d"], dtype=torch.float32, device="cuda")
        A[row, col.long()] = val
        p = _exact_dense(dict(case, kind="dual"), A, y, _vec(case["n"]), case["d"])
        return p
    return _exact_dense(case, *_dense(case, g))
