"""The passes around the Gram at the sizes where their tilings can go wrong, against the FP64
oracle (Algorithms 1 - 4): the rebuilds v <- c0 y0 + c1 A^T x and the row dots (a lane a column,
32 columns a warp; ragged K, fewer rows than a warp reads at a time, pending rows all recurring),
blocks of b = 17 .. 32 (the inverses by one CTA of 1024 threads), the row maxima of the packing
pass (scaled FP16), sampled rows that recur in most steps of a chain, a batch whose rounds have
more roles than CTAs, and the sparse dual's set-up (heavy features past the candidate list, past
the dense columns) and two sets of buffers instead of three.

Tolerances: FP64 and sparse problems 1e-10 and FP32 problems 1e-5 of the oracle, as for every
solve of these types; two forms of one solve that differ in the order of FP64 additions 1e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu

TOL64 = 1e-10
TOL32 = 1e-5


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
    return torch.as_tensor(np.ascontiguousarray(a)).cuda().contiguous()


def _rel(a, b):
    a = a.detach().cpu().numpy() if hasattr(a, "detach") else np.asarray(a)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _zeros(k):
    return torch.zeros(k, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("d,n", [(1, 1), (3, 31), (9, 32), (33, 33), (70, 4097), (257, 1000)])
@pytest.mark.parametrize("fp32,prec", [(False, "f64"), (True, "f64"), (True, "bf16x3")])
def test_rebuilds_and_row_dots(ctx, d, n, fp32, prec):
    """Both methods from a warm start, a rebuild after every outer step and the stopping test's
    row dots after every second."""
    rng = np.random.default_rng(d + n)
    X = rng.standard_normal((d, n)).astype(np.float32).astype(np.float64)
    y, tol = rng.standard_normal(n), TOL32 if fp32 else TOL64
    b, s, H, lam = min(2, d), 2, 6, 0.5
    for primal in (True, False):
        A = X if primal else X.T
        rows, cols = A.shape
        ld = (cols + 3) // 4 * 4 if fp32 else cols
        Ap = np.zeros((rows, ld), dtype=np.float32 if fp32 else np.float64)
        Ap[:, :cols] = A
        bb = min(b, rows)
        x0 = 0.1 * rng.standard_normal(rows)
        x, aux = _dev(x0), _zeros(cols)
        kw = dict(b=bb, s=s, H=H, lam=lam, seed=3, recompute_every=1)
        run = ctx.ca_bcd_solve if primal else ctx.ca_bdcd_solve
        size = dict(n=cols) if primal else dict(d=cols)
        run(_dev(Ap), _dev(y), x, aux, prec=prec, check_every=2, **size, **kw)
        ref = oracle.ca_bcd(X, y, lam, b=bb, s=s, H=H, seed=3, w0=x0, recompute_every=1) \
            if primal else oracle.ca_bdcd(X, y, lam, b=bb, s=s, H=H, seed=3, alpha0=x0,
                                          recompute_every=1)
        assert _rel(x, np.asarray(ref[0])) < tol and _rel(aux, np.asarray(ref[1])) < tol


@pytest.mark.parametrize("b,s", [(17, 1), (24, 3), (31, 2), (32, 1), (32, 5)])
@pytest.mark.parametrize("prec", ["f64", "3xtf32"])
def test_blocks_of_17_to_32(ctx, b, s, prec):
    m = synth.dense_primal(d=200, n=3001, cond=1e1, seed=b)
    X = np.ascontiguousarray(m.X[:, :3000]).astype(np.float32)
    y = m.y[:3000].copy()
    w, z = _zeros(200), _zeros(3000)
    ctx.ca_bcd_solve(_dev(X if prec != "f64" else X.astype(np.float64)), _dev(y), w, z, b=b, s=s,
                     H=4 * s + 1, lam=1e-2, seed=7, prec=prec)
    w_ref, z_ref = oracle.ca_bcd(X.astype(np.float64), y, 1e-2, b=b, s=s, H=4 * s + 1, seed=7)
    tol = TOL64 if prec == "f64" else TOL32
    assert _rel(w, w_ref) < tol and _rel(z, z_ref) < tol


@pytest.mark.parametrize("d,n", [(17, 1000), (130, 2053), (300, 8192)])
def test_row_maxima_of_the_packing_pass(ctx, d, n):
    """Scaled FP16: the row multipliers of a row-major X come from the packing pass, those of
    packed panels from a pass of their own; the padding columns of X are not part of it."""
    rng = np.random.default_rng(n)
    X = (rng.standard_normal((d, n)) * 10.0 ** rng.uniform(-3, 3, (d, 1))).astype(np.float32)
    X[d // 2] = 0.0
    y = rng.standard_normal(n)
    ld = (n + 3) // 4 * 4
    Xp = np.full((d, ld), 1e30, dtype=np.float32)
    Xp[:, :n] = X
    Xd = _dev(Xp)
    P = torch.empty(((n + 31) // 32 * d * 32,), dtype=torch.float32, device="cuda")
    ctx.ca_pack_panels(_dev(np.pad(X, ((0, 0), (0, ld - n)))), P, K=n)
    kw = dict(b=8, s=4, H=32, lam=1e-1, seed=2, prec="fp16_scaled")
    w1, z1, w2, z2 = _zeros(d), _zeros(n), _zeros(d), _zeros(n)
    ctx.ca_bcd_solve(Xd, _dev(y), w1, z1, n=n, **kw)
    ctx.ca_bcd_solve(P, _dev(y), w2, z2, panels=(d, n), **kw)
    assert torch.isfinite(w1).all() and torch.isfinite(z1).all()
    assert _rel(w1, w2.cpu().numpy()) < 1e-12 and _rel(z1, z2.cpu().numpy()) < 1e-12


@pytest.mark.parametrize("persistent", [True, False])
@pytest.mark.parametrize("N,b,s", [(10, 8, 16), (20, 4, 32), (40, 16, 8), (33, 32, 4)])
def test_chain_with_recurring_rows(ctx, N, b, s, persistent):
    rng = np.random.default_rng(N)
    X = rng.standard_normal((N, 6016)).astype(np.float32)
    y = rng.standard_normal(6016)
    w, z = _zeros(N), _zeros(6016)
    ctx.ca_set_tuning(persistent=persistent)
    ctx.ca_bcd_solve(_dev(X), _dev(y), w, z, b=b, s=s, H=3 * s + 1, lam=1.0, seed=1, prec="bf16x3")
    ctx.ca_set_tuning(persistent=True)
    w_ref, z_ref = oracle.ca_bcd(X.astype(np.float64), y, 1.0, b=b, s=s, H=3 * s + 1, seed=1)
    assert _rel(w, w_ref) < TOL32 and _rel(z, z_ref) < TOL32


def test_batch_with_more_roles_than_ctas(ctx):
    """Twelve problems of s*b = 128: each round's reduction takes several entries a CTA."""
    import paper_1612_04003_gb300 as ca
    probs, refs = [], []
    for i in range(12):
        m = synth.dense_primal(d=160 + 8 * i, n=2000 + 33 * i, cond=1e1, seed=i)
        n = (2000 + 33 * i) // 4 * 4
        X, y = np.ascontiguousarray(m.X[:, :n]).astype(np.float32), m.y[:n].copy()
        H = 32 + i
        probs.append(dict(method="primal", X=_dev(X), y=_dev(y), x=_zeros(X.shape[0]),
                          aux=_zeros(n), b=8, s=16, H=H, lam=1e-2, seed=i, prec="bf16x3"))
        refs.append(oracle.ca_bcd(X.astype(np.float64), y, 1e-2, b=8, s=16, H=H, seed=i))
    for p, r, ref in zip(probs, ctx.ca_batch_solve(probs), refs):
        assert r["status"] == ca.CA_OK and r["h_done"] == p["H"]
        assert _rel(p["x"], ref[0]) < TOL32 and _rel(p["aux"], ref[1]) < TOL32


def _csr(n, d, dens, seed):
    rng = np.random.default_rng(seed)
    mask = rng.random((n, d)) < dens[None, :]
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum(mask.sum(axis=1))
    col = np.nonzero(mask)[1].astype(np.int32)
    return rowptr, col, rng.standard_normal(len(col)).astype(np.float32), \
        np.sign(rng.standard_normal(n))


def _csr_solve(c, prob, d, **kw):
    rowptr, col, val, y = prob
    a, w = _zeros(len(y)), _zeros(d)
    c.ca_bdcd_solve((_dev(rowptr), _dev(col), _dev(val)), _dev(y), a, w, d=d, **kw)
    return a, w


@pytest.mark.parametrize("n,d,heavy", [(300, 64, 64), (300, 2, 2), (200, 1400, 650),
                                       (260, 1400, 512), (300, 1500, 3), (40, 5000, 0)])
def test_sparse_set_up(ctx, n, d, heavy):
    """Every feature heavy (more than the candidate list holds), more heavy features than dense
    columns, as many, a few, none."""
    prob = _csr(n, d, np.concatenate([np.full(heavy, 0.6), np.full(d - heavy, 0.01)]), n + d)
    kw = dict(b=8, s=8, H=40, lam=1e-1, seed=5)
    a, w = _csr_solve(ctx, prob, d, **kw)
    A = oracle.CSR(prob[0], prob[1], prob[2].astype(np.float64), d)
    a_ref, w_ref = oracle.ca_bdcd(A, prob[3], 1e-1, b=8, s=8, H=40, seed=5)
    assert _rel(a, a_ref) < TOL64 and _rel(w, w_ref) < TOL64


def test_sparse_at_a_scratch_bound(ctx):
    """The smallest bound a solve accepts, in steps smaller than a third set of Gram buffers (two
    are used there): the same result, and what is refused below it is CA_ERR_OOM."""
    import paper_1612_04003_gb300 as ca
    n, d = 700, 3000
    prob = _csr(n, d, np.full(d, 0.02), 4)
    kw = dict(b=8, s=32, H=200, lam=1e-1, seed=5)
    a_ref, w_ref = _csr_solve(ctx, prob, d, **kw)
    for bound in range(1 << 20, 64 << 20, 1 << 19):
        c = ca.Context(0, scratch_bytes_max=bound)
        try:
            a, w = _csr_solve(c, prob, d, **kw)
            break
        except ca.CaError as e:
            assert e.status == ca.CA_ERR_OOM
        finally:
            c.close()
    else:
        pytest.fail("no bound accepted")
    assert bound > 1 << 20
    assert _rel(a, a_ref.cpu().numpy()) < TOL64 and _rel(w, w_ref.cpu().numpy()) < TOL64


def test_fp64_gram_at_a_scratch_bound(ctx):
    """128 rows: 16 MB hold two partials per SM and three 64 x 64 tiles, not one per SM (2^-52 K
    m_i m_j as without a bound); 8 MB hold neither."""
    import paper_1612_04003_gb300 as ca
    rng = np.random.default_rng(2)
    A, v = rng.standard_normal((128, 9001)), rng.standard_normal(9001)
    idx = torch.arange(128, dtype=torch.int32, device="cuda")
    G = torch.empty(128, 128, dtype=torch.float64, device="cuda")
    p = torch.empty(128, dtype=torch.float64, device="cuda")
    c = ca.Context(0, scratch_bytes_max=16 << 20)
    c.ca_gram_project(_dev(A), idx, _dev(v), G, p, prec="f64")
    c.close()
    m = np.abs(A).max(1)
    Y = A.astype(np.longdouble)
    assert (np.abs(G.cpu().numpy() - Y @ Y.T) <= 2.0 ** -52 * 9001 * np.outer(m, m)).all()
    assert (np.abs(p.cpu().numpy() - Y @ v) <= 2.0 ** -52 * 9001 * m * np.abs(v).max()).all()
    c = ca.Context(0, scratch_bytes_max=8 << 20)
    with pytest.raises(ca.CaError) as e:
        c.ca_gram_project(_dev(A), idx, _dev(v), G, p, prec="f64")
    c.close()
    assert e.value.status == ca.CA_ERR_OOM


@pytest.mark.parametrize("rows,K", [(129, 1), (191, 3000), (192, 40), (193, 999), (256, 2401),
                                    (300, 33), (700, 200)])
def test_fp64_gram_of_row_pairs(ctx, rows, K):
    """More than 128 rows: pairs of groups of 64, the last one ragged; rows of magnitudes 1e-6 ..
    1e6, one group with a row outside the digits' exponent range (plain FP64 sums), one with an
    infinity.  2^-52 K m_i m_j, as for up to 128 rows, and K 2^-1074 where the square of the
    small row is a subnormal number."""
    rng = np.random.default_rng(rows)
    A = rng.standard_normal((rows, K)) * 10.0 ** rng.uniform(-6, 6, (rows, 1))
    A[70] *= 1e-160
    A[rows - 1, K // 2] = np.inf
    v = rng.standard_normal(K)
    idx = rng.permutation(rows).astype(np.int32)
    G = torch.full((rows, rows), 7.0, dtype=torch.float64, device="cuda")
    p = torch.empty(rows, dtype=torch.float64, device="cuda")
    ctx.ca_gram_project(_dev(A), _dev(idx), _dev(v), G, p, prec="f64")
    g, h, keep = G.cpu().numpy(), p.cpu().numpy(), np.isfinite(A[idx]).all(1)
    Y = A[idx][keep].astype(np.longdouble)
    m = np.abs(A[idx][keep]).max(1)
    assert (g == g.T)[np.ix_(keep, keep)].all() and not np.isfinite(g[~keep]).any()
    tol = 2.0 ** -52 * K * np.outer(m, m) + K * 2.0 ** -1074
    assert (np.abs(g[np.ix_(keep, keep)] - Y @ Y.T) <= tol).all()
    assert (np.abs(h[keep] - Y @ v) <= 2.0 ** -52 * K * m * np.abs(v).max()).all()
    assert not np.isfinite(h[~keep]).any()


@pytest.mark.parametrize("b,s", [(16, 16), (16, 9), (32, 5), (8, 40)])
def test_fp64_solve_of_row_pairs(ctx, b, s):
    """The same in a solve whose last step is short (fewer groups, or one CTA's rows)."""
    p = synth.tiny_primal(d=300, n=2001, seed=s)
    w, z = _zeros(300), _zeros(2001)
    H = 3 * s + s // 2 + 1
    ctx.ca_bcd_solve(_dev(p.X), _dev(p.y), w, z, b=b, s=s, H=H, lam=1e-1, seed=4, prec="f64")
    w_ref, z_ref = oracle.ca_bcd(p.X, p.y, 1e-1, b=b, s=s, H=H, seed=4)
    assert _rel(w, w_ref) < TOL64 and _rel(z, z_ref) < TOL64
