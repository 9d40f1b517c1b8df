"""A kept flip leaves the objective and ports that pngf_score_flips gave for it, to the
bit: both form the pivot alike."""
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


@pytest.mark.parametrize("noalloc", [False, True])
def test_accepted_objective_is_the_scored_one(P, noalloc):
    case = W.get_case("fdfd64")
    ctx = P.DbsContext(case)
    ctx.factor(W.random_design(case.n_d, 7))
    for k in np.random.default_rng(1).permutation(case.n_d)[:40]:
        f, o = ctx.score_flips([int(k)], want_ports=True)
        (P.pngf_accept_flip_noalloc if noalloc else P.pngf_accept_flip)(ctx.ctx, int(k))
        o2, f2 = ctx.eval_ports()
        assert f2 == f[0] and np.array_equal(np.ravel(o2), np.ravel(o))
    ctx.close()
