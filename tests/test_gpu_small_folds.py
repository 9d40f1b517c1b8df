"""Folds of one to eight kept flips, summed entry by entry (every kept flip of a
perfect-conductor region, batches refreshed every few flips, regions of up to 512
pixels), against a solve of the final design: the systems and the bar (1e-12) of
test_gpu_delayed.py."""
import numpy as np
import pytest

from paper_2501_18054_gb300 import workloads as W
from test_gpu_delayed import _case, _solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2501_18054_gb300 import build as B
    B.build()
    from paper_2501_18054_gb300 import pngf
    return pngf


@pytest.mark.parametrize("refresh_k", [1, 2, 3, 8, 9])
@pytest.mark.parametrize("sizes", [(1, 5, 97, 128, 129), (340, 512, 513, 100)])
def test_batch_and_solo(P, sizes, refresh_k):
    ctxs, cases = [], [_case(n, 7 * n + i, 1 + i % 3) for i, n in enumerate(sizes)]
    for i, case in enumerate(cases):
        ctxs.append(P.DbsContext(case, tau=1e-9, refresh_k=refresh_k))
        ctxs[-1].factor(W.random_design(case.n_d, i))
    P.DbsBatch(ctxs).dbs_sweep(2)
    for i, (c, case) in enumerate(zip(ctxs, cases)):
        s = P.DbsContext(case, tau=1e-9, refresh_k=refresh_k)
        s.factor(W.random_design(case.n_d, i))
        s.dbs_sweep(2)
        assert np.array_equal(c.design(), s.design())
        Wm, e, T, o = _solve(case, c.design())
        iu = np.triu_indices(case.n_d)
        for ctx in (c, s):
            st = ctx.state(with_W=True)
            for x, z in [(st["diag"], np.diag(Wm)), (st["e"], e), (st["T"], T), (st["W"][iu], Wm[iu]), (ctx.eval_ports()[0], o)]:
                assert np.max(np.abs(x - z)) <= 1e-12 * np.max(np.abs(z))
        s.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("n", [1, 6, 100, 345])
def test_single_flips_of_a_perfect_conductor_region(P, n):
    case = _case(n, 5 * n, 2)
    case.G_dd[:] += np.eye(n)  # pivots near one
    ctx = P.DbsContext(case, precision=P.PNGF_PEC)
    b = W.random_design(n, 1)
    ctx.factor(b)
    for k in [0, n // 2, 0, n - 1, n // 3]:
        ctx.accept_flip(k)
        b[k] ^= 1
        m, iu = np.flatnonzero(b), np.triu_indices(n)
        Wp = case.G_dd - case.G_dd[:, m] @ np.linalg.solve(case.G_dd[np.ix_(m, m)], case.G_dd[m, :])
        got = ctx.state(with_W=True)["W"]
        assert np.max(np.abs(got[iu] - Wp[iu])) <= 1e-12 * np.max(np.abs(case.G_dd))
        assert np.array_equal(ctx.design(), b)
    ctx.close()
