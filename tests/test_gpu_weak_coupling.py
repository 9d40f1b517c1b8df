"""Two parts of a region that hardly couple: the block of W between them keeps the
accuracy of an FP64 chain relative to its own entries, not only to the largest
entries of W (what a flip in one part does to the other is read from it).

Systems of norm below 1/2, the coupling attenuated by 1e-3 ... 1e-9.  The
reference eliminates one part after the other in 64 bits, so that every term of
the coupling block carries the attenuation.  Rounding: some 300 terms or updates
of 2**-53 with norms below 10, relative to the block's largest entry: < 1e-12.
"""
import numpy as np
import pytest

from paper_2501_18054_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2501_18054_gb300 import build as B
    B.build()
    from paper_2501_18054_gb300 import pngf
    return pngf


def _case(n, att, interleaved):
    rng = np.random.default_rng([n, int(interleaved)])
    cx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    part = np.arange(n) % 2 if interleaved else (np.arange(n) >= n // 2).astype(int)
    G = cx(n, n)
    G = (G + G.T) * np.where(part[:, None] == part[None, :], 1.0, att)
    G *= 0.3 / np.linalg.norm(G, 2)
    case = W.Case("weak", np.ascontiguousarray(G), cx(2, n), cx(n), cx(2), 1.0 + 0.3 * cx(n), np.zeros(2, complex),
                  np.ones(2, complex), W.OBJ_MAX_WEIGHTED_POWER, np.ones(2), {})
    return case, part


def _coupling_block(case, part, b):
    p, q = np.flatnonzero(part == 0), np.flatnonzero(part == 1)
    G, v = case.G_dd, case.dv * b
    blk = lambda i, j: G[np.ix_(i, j)]  # noqa: E731
    M = lambda i, j: (np.eye(len(i)) if i is j else 0.0) - blk(i, j) * v[j][None, :]  # noqa: E731
    Wq = np.linalg.solve(M(q, q), blk(q, q))  # part 1 by itself
    S = M(p, p) - M(p, q) @ np.linalg.solve(M(q, q), M(q, p))
    return np.ix_(p, q), np.linalg.solve(S, blk(p, q) - M(p, q) @ Wq)


def _check(W_upper, ix, ref):
    full = np.triu(W_upper) + np.triu(W_upper, 1).T
    assert np.max(np.abs(full[ix] - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("att", [1e-3, 1e-6, 1e-9])
def test_factor_and_search(P, att, interleaved):
    case, part = _case(290, att, interleaved)
    ctx = P.DbsContext(case, tau=1e-9, refresh_k=0)
    b = W.random_design(case.n_d, 3)
    ctx.factor(b)
    _check(ctx.state(with_W=True)["W"], *_coupling_block(case, part, b))
    assert len(ctx.dbs_sweep(3)["trace"]) > 64
    _check(ctx.state(with_W=True)["W"], *_coupling_block(case, part, ctx.design()))
    ctx.close()


@pytest.mark.parametrize("att", [1e-3, 1e-6, 1e-9])
def test_perfect_conductor(P, att):
    case, part = _case(290, att, True)
    case.G_dd[:] += np.eye(case.n_d)  # pivots near one
    ctx = P.DbsContext(case, precision=P.PNGF_PEC)
    b = W.random_design(case.n_d, 4)
    ctx.factor(b)
    Wp = case.G_dd.copy()
    for side in (0, 1):  # one part's metal after the other's
        m = np.flatnonzero((part == side) & (b == 1))
        Wp = Wp - Wp[:, m] @ np.linalg.solve(Wp[np.ix_(m, m)], Wp[m, :])
    off = [np.flatnonzero((part == s) & (b == 0)) for s in (0, 1)]
    ix = np.ix_(*off)
    _check(ctx.state(with_W=True)["W"], ix, Wp[ix])
    ctx.close()
