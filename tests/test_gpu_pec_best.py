"""Perfect-conductor search in BEST mode over several CTAs: every step keeps the
flip that scoring all pixels of the same state finds (largest gain, ties to the
lowest pixel), and ends where none clears the threshold.

The steps are driven from the host with pngf_score_flips and pngf_accept_flip on a
second context.  Both hold the state to a few thousand roundings of 2**-53 (norms
below 100), so decisions are compared while the best two gains and the
threshold differ by more than 1e-9 |f|, the values to 1e-9.
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


@pytest.mark.parametrize("side,n_ctas", [(16, 0), (21, 0), (21, 2), (32, 0)])
def test_pec_best_equals_host_driven_steps(P, side, n_ctas):
    big = W.get_case("fdfd128_metal")
    x0 = (32 - side) // 2
    case = big.sub_case([(x0 + i) * 32 + x0 + j for i in range(side) for j in range(side)])
    n, steps, tau = case.n_d, 40, 1e-6
    b0 = W.random_design(n, side)
    host, dev = (P.DbsContext(case, precision=P.PNGF_PEC, mode=P.PNGF_BEST_IMPROVEMENT, tau=tau, n_ctas=n_ctas) for _ in range(2))
    host.factor(b0)
    dev.factor(b0)
    res = dev.dbs_sweep(steps)
    sign = 1.0 if case.obj_kind == W.OBJ_MAX_WEIGHTED_POWER else -1.0
    f = host.eval_ports()[1]
    for i in range(steps):
        gain = sign * (host.score_flips(np.arange(n)) - f)
        gain = np.where(np.isnan(gain), -np.inf, gain)
        k = int(np.argmax(gain))
        second = np.partition(gain, -2)[-2]
        if min(abs(gain[k] - tau * abs(f)), gain[k] - second) < 1e-9 * abs(f):
            break
        if gain[k] <= tau * abs(f):
            assert len(res["trace"]) == i and res["counters"][3] == 1
            break
        assert tuple(int(v) for v in res["trace"][i][:3]) == (i, 0, k)
        host.accept_flip(k)
        f = host.eval_ports()[1]
        assert abs(res["trace_f"][i] - f) <= 1e-9 * abs(f)
    else:
        assert len(res["trace"]) == steps and np.array_equal(dev.design(), host.design())
    assert i >= 5
    host.close()
    dev.close()
