"""Digit products where a row's largest entry is just below a power of two (its
leading digit rounds up, the scale moves on by one) and far above the rest.

The entries of G at pixels that are off against pixels that are on are operands
as they are (dv = 1); each such row's largest one is a fraction c of a power of two,
of either sign, in its real or imaginary part.  Norm of G below 1/2: two correct FP64
solvers agree to 1e-12, as in test_gpu_factor.py.
"""
import numpy as np
import pytest

from paper_2501_18054_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FRACTIONS = [1 - 2.0**-53, 1 - 2.0**-20, 1 - 2.0**-9, 1 - 2.0**-8, 1 - 2.0**-8 - 2.0**-20, 127.49805 / 128, 127.498 / 128,
             127.49 / 128, 127.47 / 128, 127.4 / 128, 0.5, 0.5 + 2.0**-53]


@pytest.fixture(scope="module")
def P():
    from paper_2501_18054_gb300 import build as B
    B.build()
    from paper_2501_18054_gb300 import pngf
    return pngf


def test_factor_with_largest_entries_near_a_power_of_two(P):
    n, rng = 192, np.random.default_rng(9)
    cx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    G = cx(n, n) * 2.0**-9
    G = G + G.T
    on = np.sort(rng.permutation(n)[:n // 2])
    off = np.setdiff1d(np.arange(n), on)
    for q, i in enumerate(off):
        v = FRACTIONS[q % len(FRACTIONS)] * 2.0**-4 * (1, -1, 1j, -1j)[q // len(FRACTIONS) % 4]
        G[i, on[q]] = G[on[q], i] = v
    case = W.Case("scale", np.ascontiguousarray(G), cx(2, n), cx(n), cx(2), np.ones(n, complex), np.zeros(2, complex),
                  np.ones(2, complex), W.OBJ_MAX_WEIGHTED_POWER, np.ones(2), {})
    b = np.zeros(n, np.uint8)
    b[on] = 1
    ctx = P.DbsContext(case, tau=1e-9, refresh_k=0)
    ctx.factor(b)
    for _ in range(2):  # the factor, then a search whose folds digitise columns of W
        st, b = ctx.state(with_W=True), ctx.design()
        M = np.eye(n) - G * b[None, :]
        Wm, iu = np.linalg.solve(M, G), np.triu_indices(n)
        assert np.max(np.abs(st["W"][iu] - Wm[iu])) <= 1e-12 * np.max(np.abs(Wm))
        assert np.max(np.abs(st["e"] - np.linalg.solve(M, case.c_d))) <= 1e-12 * np.max(np.abs(st["e"]))
        ctx.dbs_sweep(2)
    ctx.close()
