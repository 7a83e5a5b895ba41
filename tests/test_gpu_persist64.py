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
    ("primal", 40, 17, 1, 1, 23, 0, 0),
    ("primal", 64, 1024, 4, 4, 202, 0, 0),
    ("primal", 33, 1057, 8, 4, 61, 4, 0),
    ("primal", 60, 5003, 16, 2, 31, 0, 3),
    ("dual", 4832, 48, 8, 3, 40, 0, 0),
    ("dual", 31, 200, 16, 1, 37, 5, 0),
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
