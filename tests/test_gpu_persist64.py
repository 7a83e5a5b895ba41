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


def _uneven(rng, rows, K, kind):
    """Rows whose entries of G are far below the product of the two rows' largest magnitudes."""
    A = rng.standard_normal((rows, K))
    if kind == "spikes":  # one large element a row, in different columns
        A[np.arange(rows), rng.permutation(max(rows, K))[:rows] % K] *= 1e9
    elif kind == "one":  # one such row
        A[rows // 2, K // 2] *= 1e9
    elif kind == "spread":  # elements of any magnitude
        A *= 10.0 ** rng.uniform(-12, 12, (rows, K))
    elif kind == "supports":  # a few nonzero columns a row, and a tiny one that all rows share
        A *= rng.random((rows, K)) < 0.1
        A[:, K // 3] = 1e-9 * (1.0 + rng.random(rows))
    elif kind == "groups":  # groups of columns in units of their own, each row at home in one
        unit = 10.0 ** rng.uniform(-8, 8, 4)
        home = rng.integers(0, 4, rows)
        A *= np.where(np.arange(K)[None] % 4 == home[:, None], unit[home][:, None], 1e-10)
    return A


@pytest.mark.parametrize("kind", ["even", "spikes", "one", "spread", "supports", "groups"])
@pytest.mark.parametrize("rows,K", [(16, 180), (17, 31), (32, 4000), (33, 180), (64, 5003),
                                    (100, 16), (128, 180), (20, 30011),
                                    (40, 30011), (128, 30011), (200, 700), (300, 5003)])
def test_fp64_gram_entry_by_entry(ctx, rows, K, kind):
    """G = Y Y^T of FP64 rows, every entry against its own terms: S_ij = sum |y_ik y_jk|.  A segment
    of n <= 192 columns is within 1.2 x 128 or (n > 128) n 2^-53 S; the sums of a CTA's
    segments, of the at most 152 partials and the last rounding add one 2^-53 S each; K <= 30011
    gives a CTA two segments, or (row pairs, K <= 5003) nine on at least four CTAs."""
    rng = np.random.default_rng(rows * 7 + K)
    A = _uneven(rng, rows, K, kind)
    v = rng.standard_normal(K)
    G = torch.empty(rows, rows, dtype=torch.float64, device="cuda")
    p = torch.empty(rows, dtype=torch.float64, device="cuda")
    idx = rng.permutation(rows).astype(np.int32)
    ctx.ca_gram_project(_dev(A), _dev(idx), _dev(v), G, p, prec="f64")
    cols = np.sort(rng.permutation(rows)[:24])  # (extended precision is slow: 24 columns of G)
    Y = A[idx].astype(np.longdouble)
    S = np.abs(Y) @ np.abs(Y[cols]).T
    g = G.cpu().numpy()
    assert (g == g.T).all()
    assert (np.abs(g[:, cols] - Y @ Y[cols].T) <= 2.0 ** -53 * (198 + 9 + 152 + 1) * S).all()


@pytest.mark.parametrize("rows", [20, 70])
def test_fp64_gram_zero_rows_and_infinities(ctx, rows):
    """A row of zeros loses nothing to digits, but times an infinity or a NaN it is a NaN."""
    rng = np.random.default_rng(4)
    A = rng.standard_normal((rows, 700))
    A[2], A[3, 100:400] = 0.0, 0.0
    A[5, 120], A[7, 20], A[9] = -np.inf, np.nan, 1e-310
    G = torch.empty(rows, rows, dtype=torch.float64, device="cuda")
    p = torch.empty(rows, dtype=torch.float64, device="cuda")
    ctx.ca_gram_project(_dev(A), torch.arange(rows, dtype=torch.int32, device="cuda"),
                        _dev(rng.standard_normal(700)), G, p, prec="f64")
    g = G.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = (A[:, None] * A[None]).sum(-1)
        S = (np.abs(A[:, None]) * np.abs(A[None])).sum(-1)
    assert (np.isnan(g) == np.isnan(ref)).all() and (np.isinf(g) == np.isinf(ref)).all()
    fin = np.isfinite(ref)
    # (numpy's pairwise sum and ours; products with the small row round to 2^-1075 each)
    assert (np.abs(g[fin] - ref[fin]) <= 2.0 ** -53 * 700 * S[fin] + 700 * 2.0 ** -1074).all()


@pytest.mark.parametrize("method,d,n,b,s", [("primal", 6, 70, 1, 1), ("dual", 40, 9, 2, 1)])
def test_more_steps_than_a_launch(ctx, method, d, n, b, s):
    """65536 steps go to one launch; the update of its last one is applied before the next launch."""
    p = synth.tiny_primal(d=d, n=n, seed=2)
    lam, H = 1e-1, 65536 * s + 5
    x = torch.zeros(d if method == "primal" else n, dtype=torch.float64, device="cuda")
    aux = torch.zeros(n if method == "primal" else d, dtype=torch.float64, device="cuda")
    kw = dict(b=b, s=s, H=H, seed=3)
    if method == "primal":
        ctx.ca_bcd_solve(_dev(p.X), _dev(p.y), x, aux, lam=lam, prec="f64", **kw)
        ref = oracle.ca_bcd(p.X, p.y, lam, **kw)
    else:
        ctx.ca_bdcd_solve(_dev(p.X.T), _dev(p.y), x, aux, lam=lam, prec="f64", **kw)
        ref = oracle.ca_bdcd(p.X, p.y, lam, **kw)
    assert _rel(x.cpu().numpy(), np.asarray(ref[0])) < 1e-10
    assert _rel(aux.cpu().numpy(), np.asarray(ref[1])) < 1e-10
