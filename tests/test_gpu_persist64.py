"""The persistent launch of dense FP64 outer steps (CA-BCD, Algorithm 2; CA-BDCD, Algorithm 4)
against the FP64 oracle and against one launch per kernel and step.

Sizes at its edges: fewer columns than a 32-column tile, a ragged last tile, as many tiles as
columns CTAs and more, one row a step, the largest s*b of each Gram form, a short last step, a
recomputation and a check inside the run, a warm start (a pending update never reaches the
first launch then).  Tolerances: the FP64 path's 1e-10 against the oracle; the two forms sum the
same FP64 products in other orders and solve the same double-float chain (2^-44 of a block's
condition number, below 1e3 here): 1e-10.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1612_04003_gb300 as ca
    ca.build()
    c = ca.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


CASES = [  # method, d, n, b, s, H, recompute_every, check_every
    # s*b = 16 | 17 .. 128: the Gram on CUDA cores | by digit products
    ("primal", 40, 17, 1, 1, 23, 0, 0),
    ("primal", 64, 1024, 4, 4, 202, 0, 0),
    ("primal", 33, 1057, 8, 4, 61, 4, 0),
    ("primal", 60, 5003, 16, 2, 31, 0, 3),
    ("dual", 4832, 48, 8, 3, 40, 0, 0),
    ("dual", 31, 200, 16, 1, 37, 5, 0),
    ("primal", 90, 4999, 8, 4, 41, 0, 0),
    ("dual", 1500, 90, 1, 17, 70, 0, 2),
    ("primal", 70, 33, 16, 4, 18, 0, 0),
    ("dual", 5001, 160, 16, 8, 28, 2, 0),
    ("primal", 130, 777, 8, 16, 50, 0, 0),
    ("primal", 40, 36001, 8, 5, 33, 0, 0),  # two segments of columns a CTA
]


@pytest.mark.parametrize("method,d,n,b,s,H,every,check", CASES)
def test_persistent_fp64_steps(ctx, method, d, n, b, s, H, every, check):
    p = synth.tiny_primal(d=d, n=n, seed=d + n)
    lam = 1e-1
    kw = dict(b=b, s=s, H=H, lam=lam, seed=5, prec="f64", recompute_every=every, check_every=check)
    rng = np.random.default_rng(3)
    x0 = 0.1 * rng.standard_normal(d if method == "primal" else n)
    got = []
    for persistent in (True, False):
        ctx.ca_set_tuning(persistent=persistent)
        x = _dev(x0)
        aux = torch.zeros(n if method == "primal" else d, dtype=torch.float64, device="cuda")
        if method == "primal":
            ctx.ca_bcd_solve(_dev(p.X), _dev(p.y), x, aux, **kw)
        else:
            ctx.ca_bdcd_solve(_dev(p.X.T), _dev(p.y), x, aux, **kw)
        got.append((x.cpu().numpy(), aux.cpu().numpy()))
    ctx.ca_set_tuning(persistent=True)
    if method == "primal":
        ref = oracle.ca_bcd(p.X, p.y, lam, b=b, s=s, H=H, seed=5, w0=x0, recompute_every=every)
    else:
        ref = oracle.ca_bdcd(p.X, p.y, lam, b=b, s=s, H=H, seed=5, alpha0=x0, recompute_every=every)
    for i in range(2):
        assert _rel(got[0][i], np.asarray(ref[i])) < 1e-10
        assert _rel(got[0][i], got[1][i]) < 1e-10


@pytest.mark.parametrize("rows,K,scale", [(1, 1, 0), (16, 40, 0), (17, 31, 0), (32, 4000, 0),
                                          (33, 999, 1), (64, 32, 0), (100, 5000, 1),
                                          (128, 30011, 0), (128, 70, 2)])
def test_gram_fp64(ctx, rows, K, scale):
    """G = Y Y^T and p = Y v of FP64 rows against extended precision.  Digit products: each
    element is rounded to 2^-55 of its row's largest magnitude m in the segment, the levels left
    out and the one rounded accumulator are smaller, so an entry is within 2^-52 K m_i m_j (an
    FP64 sum: 2^-53 K times the sum of |products|, about the same).  scale 1: rows of magnitudes
    1e-6 .. 1e6 and single large elements; 2: rows outside the digits' exponent range."""
    rng = np.random.default_rng(rows + K)
    A = rng.standard_normal((rows + 3, K))
    if scale == 1:
        A *= 10.0 ** rng.uniform(-6, 6, size=(rows + 3, 1))
        A[np.arange(rows), rng.integers(0, K, rows)] *= 1e9
        A[5] = 0.0
    if scale == 2:
        A *= (1e-150 ** rng.integers(0, 2, size=(rows + 3, 1)))
    idx = rng.permutation(rows + 3)[:rows].astype(np.int32)
    v = rng.standard_normal(K)
    G = torch.empty(rows, rows, dtype=torch.float64, device="cuda")
    p = torch.empty(rows, dtype=torch.float64, device="cuda")
    ctx.ca_gram_project(_dev(A), _dev(idx), _dev(v), G, p, prec="f64")
    Y = A[idx].astype(np.longdouble)
    m = np.abs(A[idx]).max(1)
    assert (np.abs(G.cpu().numpy() - Y @ Y.T) <= 2.0 ** -52 * K * np.outer(m, m)).all()
    assert (np.abs(p.cpu().numpy() - Y @ v) <= 2.0 ** -52 * K * m * np.abs(v).max()).all()


def test_gram_fp64_non_finite(ctx):
    """An infinity or a NaN in one row reaches exactly the entries FP64 arithmetic gives."""
    rng = np.random.default_rng(1)
    A = rng.standard_normal((40, 500))
    A[3, 100], A[7, 20] = np.inf, np.nan
    G = torch.empty(40, 40, dtype=torch.float64, device="cuda")
    p = torch.empty(40, dtype=torch.float64, device="cuda")
    ctx.ca_gram_project(_dev(A), torch.arange(40, dtype=torch.int32, device="cuda"),
                        _dev(rng.standard_normal(500)), G, p, prec="f64")
    g, ref = G.cpu().numpy(), A @ A.T
    assert (np.isnan(g) == np.isnan(ref)).all() and (np.isinf(g) == np.isinf(ref)).all()
    fin = np.isfinite(ref)
    assert np.abs(g[fin] - ref[fin]).max() <= 2.0 ** -52 * 500 * 25


@pytest.mark.parametrize("method,d,n,b,s", [("primal", 150, 2003, 7, 17), ("dual", 2003, 150, 7, 18),
                                            ("primal", 140, 999, 5, 25), ("dual", 700, 140, 3, 42)])
def test_odd_blocks_in_turn(ctx, method, d, n, b, s):
    """Odd b with more than 16 blocks a step: an inverse CTA takes several blocks one after another,
    and the last pivot of one and the first of the next are both even.  Seven steps, the last one
    short; 1e-10, as for every FP64 solve."""
    p = synth.tiny_primal(d=d, n=n, seed=b + s)
    lam, H = 1e-1, 6 * s + 5
    x = torch.zeros(d if method == "primal" else n, dtype=torch.float64, device="cuda")
    aux = torch.zeros(n if method == "primal" else d, dtype=torch.float64, device="cuda")
    kw = dict(b=b, s=s, H=H, seed=9)
    if method == "primal":
        ctx.ca_bcd_solve(_dev(p.X), _dev(p.y), x, aux, lam=lam, prec="f64", **kw)
        ref = oracle.ca_bcd(p.X, p.y, lam, **kw)
    else:
        ctx.ca_bdcd_solve(_dev(p.X.T), _dev(p.y), x, aux, lam=lam, prec="f64", **kw)
        ref = oracle.ca_bdcd(p.X, p.y, lam, **kw)
    assert _rel(x.cpu().numpy(), np.asarray(ref[0])) < 1e-10
    assert _rel(aux.cpu().numpy(), np.asarray(ref[1])) < 1e-10
