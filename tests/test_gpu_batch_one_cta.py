"""FP64 batches, above all with one CTA per run: regions of more than one scoring chunk (128
positions), folds of more than one row block (128 rows) inside a sweep, the
refresh of a whole run by one CTA, and regions above 1024 pixels.

A run of fewer than four pixels, or one above 1024, keeps the whole batch on one
CTA per run.  Every run is compared with the same run done alone, bit for bit
without refreshes (the same arithmetic) and to 1e-12 with them (the ports and
corrections of a refresh are summed in another order: 2**-53 times the terms'
number), and its final state with a solve of its final design (1e-12, the bound
of test_gpu_delayed.py for the same systems).  Many chunks hold no improving flip
(late sweeps), many sweeps end with an empty delayed set.
"""
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


@pytest.mark.parametrize("refresh_k", [0, 64])
@pytest.mark.parametrize("sizes", [(130, 3, 300, 257, 128), (1030, 129)])
def test_one_cta_batch_equals_solo(P, sizes, refresh_k):
    sweeps = 6
    runs = []
    for i, n in enumerate(sizes):
        runs.append((_case(n, 13 * n + i, 1 + i % 3), W.random_design(n, i), W.shuffled_order(n, sweeps, seed=i) if i % 2 == 0 else None))

    def context(case, b):
        c = P.DbsContext(case, tau=1e-9, refresh_k=refresh_k)
        c.factor(b)
        return c

    ctxs = [context(case, b) for case, b, _ in runs]
    res = P.DbsBatch(ctxs).dbs_sweep(sweeps, orders=[o for _, _, o in runs])
    for c, r, (case, b, order) in zip(ctxs, res, runs):
        s = context(case, b)
        rs = s.dbs_sweep(sweeps, order=order)
        assert np.array_equal(r["trace"], rs["trace"]) and np.array_equal(c.design(), s.design())
        assert np.array_equal(r["counters"][:7], rs["counters"][:7])
        if case.n_d > 256:
            assert np.bincount(r["trace"][:, 0]).max() > 64  # folds inside a sweep
        a, e = c.state(with_W=True), s.state(with_W=True)
        Wm, ex, T, o = _solve(case, c.design())
        iu = np.triu_indices(case.n_d)
        for x, y, z in [(a["diag"], e["diag"], np.diag(Wm)), (a["e"], e["e"], ex), (a["T"], e["T"], T),
                        (a["W"][iu], e["W"][iu], Wm[iu]), (c.eval_ports()[0], s.eval_ports()[0], o)]:
            bar = 1e-12 * np.max(np.abs(z))
            assert np.max(np.abs(x - z)) <= bar
            assert np.array_equal(x, y) if refresh_k == 0 else np.max(np.abs(x - y)) <= bar
        s.close()
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("sizes", [(600, 257, 300)])
def test_cluster_batch_of_larger_regions(P, sizes):
    """Few large runs, on clusters: shares of more than 64 pixels, whose delayed
    columns are read from global memory; W against a solve."""
    ctxs, cases = [], [_case(n, 5 * n + i, 1 + i) for i, n in enumerate(sizes)]
    for i, case in enumerate(cases):
        ctxs.append(P.DbsContext(case, tau=1e-9, refresh_k=50))
        ctxs[-1].factor(W.random_design(case.n_d, i))
    for c, case, r in zip(ctxs, cases, P.DbsBatch(ctxs).dbs_sweep(4)):
        assert len(r["trace"]) > 64
        Wm, e, T, o = _solve(case, c.design())
        st, iu = c.state(with_W=True), np.triu_indices(case.n_d)
        for x, z in [(st["diag"], np.diag(Wm)), (st["e"], e), (st["T"], T), (st["W"][iu], Wm[iu]), (c.eval_ports()[0], o)]:
            assert np.max(np.abs(x - z)) <= 1e-12 * np.max(np.abs(z))
        c.close()


@pytest.mark.parametrize("sizes,other", [((100, 97, 64), 3), ((300, 120), 3), ((150, 300), 1030)])
def test_a_run_does_not_depend_on_the_batch_around_it(P, sizes, other):
    """The same runs on clusters, and on one CTA each (sent there by one more run),
    with refreshes: the same bits."""
    def batch(extra):
        ctxs, orders = [], []
        for i, n in enumerate(list(sizes) + extra):
            c = P.DbsContext(_case(n, 3 * n + i, 1 + i % 3), tau=1e-9, refresh_k=5)
            c.factor(W.random_design(n, i))
            ctxs.append(c)
            orders.append(W.shuffled_order(n, 3, seed=i) if i % 2 else None)
        res = P.DbsBatch(ctxs).dbs_sweep(3, orders=orders)
        out = [(r["trace"], r["trace_f"], r["counters"], c.state(with_W=True), c.eval_ports(), c.design()) for c, r in zip(ctxs, res)]
        for c in ctxs:
            c.close()
        return out

    for a, b, n in zip(batch([]), batch([other]), sizes):
        iu = np.triu_indices(n)
        for x, y in zip(a[:3], b[:3]):
            assert np.array_equal(x, y)
        for key in ("diag", "e", "T"):
            assert np.array_equal(a[3][key], b[3][key])
        assert np.array_equal(a[3]["W"][iu], b[3]["W"][iu])
        assert np.array_equal(a[4][0], b[4][0]) and a[4][1] == b[4][1] and np.array_equal(a[5], b[5])
        assert a[2][4] > 2  # refreshes
