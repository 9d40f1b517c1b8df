"""FP64 batches whose large runs are few, advanced by clusters of CTAs: every run
ends as the same run done alone, at the smallest and ragged regions (fewer
pixels than a warp, shares of unequal size) and with explicit visiting orders.

Without refreshes a search is the same arithmetic whatever the CTAs that share
it, so traces, designs, ports and state are equal bit for bit.  A refresh sums the
ports over the CTAs' partial sums in another order and corrects e and T to the
residual's rounding: 1e-12 of the largest value (2**-53 times the ~100 terms and a
few units of conditioning), with the same kept flips.
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


@pytest.mark.parametrize("refresh_k", [0, 5])
@pytest.mark.parametrize("sizes", [(100, 4, 33), (97, 64, 5, 31), (100,) * 9])
def test_cluster_batch_equals_solo(P, sizes, refresh_k):
    case = W.get_case("fdfd64")
    rng = np.random.default_rng(5)
    runs = []
    for i, n in enumerate(sizes):
        sub = case if n == 100 else case.sub_case(np.sort(rng.choice(100, n, False)))
        order = W.shuffled_order(n, 4, seed=i) if i % 2 else None
        runs.append((sub, W.random_design(n, i), order))

    def context(sub, b):
        c = P.DbsContext(sub, precision=P.PNGF_FP64, tau=1e-9, refresh_k=refresh_k)
        c.factor(b)
        return c

    ctxs = [context(sub, b) for sub, b, _ in runs]
    res = P.DbsBatch(ctxs).dbs_sweep(4, orders=[o for _, _, o in runs])
    for c, r, (sub, b, order) in zip(ctxs, res, runs):
        s = context(sub, b)
        rs = s.dbs_sweep(4, order=order)
        assert np.array_equal(r["trace"], rs["trace"]) and np.array_equal(c.design(), s.design())
        assert np.array_equal(r["counters"][:7], rs["counters"][:7])
        a, e = c.state(with_W=True), s.state(with_W=True)
        iu = np.triu_indices(sub.n_d)
        for x, y in [(r["trace_f"], rs["trace_f"]), (a["diag"], e["diag"]), (a["e"], e["e"]), (a["T"], e["T"]),
                     (a["W"][iu], e["W"][iu]), (c.eval_ports()[0], s.eval_ports()[0])]:
            if refresh_k == 0:
                assert np.array_equal(x, y)
            else:
                assert np.max(np.abs(x - y), initial=0.0) <= 1e-12 * max(np.max(np.abs(y), initial=0.0), 1e-300)
        s.close()
    for c in ctxs:
        c.close()
