"""Entries of G that are not finite are reported by the factor wherever they stand, also
between two pixels that are off (the elimination of the whole system meets them
as a column without a pivot), and by the perfect-conductor state when its pivot is."""
import numpy as np
import pytest

from paper_2501_18054_gb300 import workloads as W
from test_gpu_delayed import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2501_18054_gb300 import build as B
    B.build()
    from paper_2501_18054_gb300 import pngf
    return pngf


@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, 1j * np.inf])
@pytest.mark.parametrize("n", [40, 150])
def test_factor_reports_a_bad_entry_anywhere(P, n, value):
    case = _case(n, n, 2)
    b = W.random_design(n, 1)
    on, off = np.flatnonzero(b), np.flatnonzero(b == 0)
    for i, j in ((off[1], off[4]), (off[3], off[3]), (on[2], off[2]), (on[1], on[5])):
        G = case.G_dd.copy()
        case.G_dd[i, j] = case.G_dd[j, i] = value
        ctx = P.DbsContext(case)
        ctx.factor(b)
        assert ctx.sync() == P.PNGF_ESINGULAR, (i, j)
        ctx.close()
        case.G_dd[:] = G


@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf])
def test_perfect_conductor_reports_a_bad_pivot(P, value):
    case = _case(60, 60, 2)
    b = W.random_design(60, 1)
    k = int(np.flatnonzero(b)[3])
    case.G_dd[k, k] = value
    ctx = P.DbsContext(case, precision=P.PNGF_PEC)
    ctx.factor(b)
    assert ctx.sync() == P.PNGF_ENUMERIC
    ctx.close()
