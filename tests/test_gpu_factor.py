"""The factor's blocked elimination at the edges of its blocks (FP64 state).

Only the m pixels that are on are eliminated (panels of 32 columns,
substitution blocks of 64 rows, product tiles of 128 x 64), so the edges are in
m and in n - m, wherever the pixels lie.  The systems are well conditioned
(||G V|| < 1/2), so two correct FP64 solvers agree to a small multiple of
n * 2^-53 < 1e-13; the bar is 1e-12.
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


def _case(n, seed, n_o=2):
    rng = np.random.default_rng(seed)
    cx = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    G = cx(n, n)
    # rows of very different magnitude: every operand row has its own scale
    s = 10.0 ** rng.uniform(-3, 0, n)
    G = (G + G.T) * s[:, None] * s[None, :]
    G *= 0.5 / max(1e-300, np.linalg.norm(G, 2)) / 2.0
    return W.Case("edge", np.ascontiguousarray(G), cx(n_o, n), cx(n), cx(n_o), cx(n) * 0.5 + 1.0, np.zeros(n_o, complex),
                  np.ones(n_o, complex), W.OBJ_MAX_WEIGHTED_POWER, np.ones(n_o), {})


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (33, 0), (33, 33), (64, 31), (65, 32), (97, 33), (130, 63), (130, 64),
                                 (131, 65), (200, 127), (300, 128), (257, 129), (400, 257)])
def test_factor_at_block_edges(P, n, m):
    case = _case(n, 7 * n + m, n_o=1 + n % 8)
    rng = np.random.default_rng(n + m)
    b = np.zeros(n, np.uint8)
    b[rng.permutation(n)[:m]] = 1
    ctx = P.DbsContext(case)
    ctx.factor(b)
    assert ctx.sync() == P.PNGF_OK
    st = ctx.state(with_W=True)
    v = case.dv * b
    M = np.eye(n) - case.G_dd * v[None, :]
    Wr = np.linalg.solve(M, case.G_dd)
    e = np.linalg.solve(M, case.c_d)
    assert _rel(st["W"], Wr) < 1e-12
    assert np.array_equal(st["W"], st["W"].T)
    assert np.array_equal(st["diag"], np.diag(st["W"]))
    assert _rel(st["e"], e) < 1e-12
    assert _rel(st["T"], case.G_od + (case.G_od * v[None, :]) @ Wr) < 1e-12
    o, _ = ctx.eval_ports()
    assert _rel(o, case.c_o + case.G_od @ (v * e)) < 1e-12
    assert np.array_equal(ctx.design(), b)
    ctx.close()


def test_singular_and_non_finite_systems_are_reported(P):
    # M = diag(1 - g_k v_k) with one pivot exactly zero
    n = 40
    case = _case(n, 3)
    case.G_dd[:] = np.diag(np.full(n, 0.5))
    case.dv[:] = 1.0
    case.dv[7] = 2.0
    ctx = P.DbsContext(case)
    ctx.factor(np.ones(n, np.uint8))
    assert ctx.sync() == P.PNGF_ESINGULAR
    b = np.ones(n, np.uint8)
    b[7] = 0  # the same system without that pixel is regular
    ctx.factor(b)
    assert ctx.sync() == P.PNGF_OK
    ctx.close()
    # a NaN in G reaches everything that depends on it
    case = _case(100, 4)
    case.G_dd[3, 5] = case.G_dd[5, 3] = np.nan
    ctx = P.DbsContext(case)
    ctx.factor(np.ones(100, np.uint8))
    ctx.sync()
    assert np.all(np.isnan(ctx.state()["e"]))
    ctx.close()
