"""The FP64 leaf TRSM by refinement (through hrp_trsm with an all-FP64 tree, leaf 128) at the edges
of its row tiles (16, 32), column groups (8, 16) and thread counts (64 columns), and where it must
hand its rows to the FP64 substitution: ill-conditioned, far outside binary32's range, NaN.

Bound: the rows of X solve X L^T = B with a backward error of FP64 substitution, per entry
|B - X L^T| <= nc 2^-53 |X| |L|^T (Higham, Thm. 8.5), the refinement's fixed point adding at most
nc 2^-58 of the row's and column's largest entries.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    yield hrp, h, torch
    h.close()


def _factor(n, kind, rng):
    if kind == "dominant":
        L = np.tril(rng.standard_normal((n, n))) / np.sqrt(n)
        L[np.arange(n), np.arange(n)] = 2 * np.sqrt(n)
        return L, np.ones(n)
    G = rng.standard_normal((n, max(1, n // 2)))
    A = G @ G.T / max(1, n // 2) + (1e-2 if kind != "ill" else 1e-9) * np.eye(n)
    d = np.ones(n)
    if kind == "graded":
        d = np.exp2(rng.integers(-150, 150, n).astype(float))
    if kind == "huge":
        d = np.full(n, 2.0 ** 200)
    return np.linalg.cholesky(A) * d[:, None], d


def _solve(env, L, B):
    hrp, h, torch = env
    Bt = hrp.colmajor(B).cuda()
    h.trsm(hrp.tree_parse("[F64]", leaf=128), hrp.colmajor(L).cuda(), Bt)
    assert h.check() == 0
    return hrp.from_colmajor(Bt)


@pytest.mark.parametrize("kind", ["dominant", "gram", "ill", "graded", "huge"])
@pytest.mark.parametrize("m,n", [(1, 32), (15, 33), (17, 64), (33, 65), (16, 100), (200, 127), (2500, 128), (2433, 40)])
def test_refined_trsm_meets_the_substitution_bound(env, m, n, kind):
    rng = np.random.default_rng(7 * m + n)
    L, d = _factor(n, kind, rng)
    B = rng.standard_normal((m, n)) * d[None, :] * np.exp2(rng.integers(-40, 40, m).astype(float))[:, None]
    X = _solve(env, L, B)
    Lq, Xq = L.astype(np.longdouble), X.astype(np.longdouble)
    res = np.abs(B.astype(np.longdouble) - Xq @ Lq.T)
    aX, aL = np.abs(Xq), np.abs(Lq)
    row = aX.max(1)
    bound = n * np.longdouble(2.0) ** -53 * (aX @ aL.T) + n * np.longdouble(2.0) ** -58 * row[:, None] * aL.sum(1)[None, :]
    assert np.all(res <= bound), float(np.max(res / bound))


def test_refined_trsm_carries_nan_in_its_row_only(env):
    rng = np.random.default_rng(3)
    L, _ = _factor(64, "gram", rng)
    B = rng.standard_normal((40, 64))
    ref = _solve(env, L, B)
    B[5, 10] = np.nan
    X = _solve(env, L, B)
    assert np.isnan(X[5, 10:]).all() and np.isfinite(X[5, :10]).all()
    keep = np.arange(40) != 5
    assert np.allclose(X[keep], ref[keep], rtol=1e-12, atol=0)
