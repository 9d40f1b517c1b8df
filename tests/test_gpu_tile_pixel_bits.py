"""Tiles of one pixel: the search (one thread per candidate) scores them with the bits of
pngf_score_tiles (one warp per candidate).

A search over one tile keeps it exactly if its gain exceeds tau |F|.  With tau two
roundings (4.5e-16) below and above the gain that pngf_score_tiles gives, the search
must keep and refuse it: the quotient, the step and the product are off by 3.3e-16
together, and a score that differs in its last bits is off by more where the gain is
a part of F."""
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


@pytest.mark.parametrize("name,side,n", [("fdfd64", 10, 10), ("fdfd128_metal", 32, 12)])
def test_search_scores_as_score_tiles(P, name, side, n):
    x0 = (side - n) // 2
    case = W.get_case(name).sub_case([(x0 + i) * side + x0 + j for i in range(n) for j in range(n)])
    b = W.random_design(case.n_d, 2)
    ctx = P.DbsContext(case)
    ctx.factor(b)
    F0 = ctx.eval_ports()[1]
    F = P.TileSearch([ctx], np.arange(case.n_d)).score(np.arange(case.n_d))
    gain = (F - F0) * (1.0 if case.obj_kind == W.OBJ_MAX_WEIGHTED_POWER else -1.0)
    picks = [k for k in np.argsort(-gain) if gain[k] > 1e-3 * abs(F0)][:40]
    assert len(picks) >= 10
    for k in picks:
        for step, kept in ((1 - 4.5e-16, 1), (1 + 4.5e-16, 0)):
            c = P.DbsContext(case, tau=gain[k] / abs(F0) * step)
            c.factor(b)
            assert len(P.TileSearch([c], [[int(k)]]).dbs_sweep(1)["trace"]) == kept, (k, step)
            c.close()
    ctx.close()
