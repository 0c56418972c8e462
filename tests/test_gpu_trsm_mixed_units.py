"""FP64 leaf TRSM by refinement whose rows or columns are in different units: an entry of X is accurate
against its own terms, whatever other rows or columns share its scales.

Bounds: substitution leaves |B - X L^T| <= n 2^-53 |X| |L|^T per entry (Higham, Thm. 8.5).  The refinement
holds a residual to 2^-59.8 of its scales (128 terms, ordinary digits) where sum |x| |l| is at least
2^-12 of them: 2^-47.8, under 4 n 2^-53 for the orders here.  A Cholesky factor leaves |A - L L^T| <=
(n + 1) 2^-53 d d^T, d_i = sqrt(a_ii) (Higham, Thm. 10.5); 4 (n + 1) 2^-53 for the same reason.
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


def _dominant(n, rng):
    B = rng.standard_normal((n, n))
    M = (B + B.T) / 2
    np.fill_diagonal(M, 0)
    np.fill_diagonal(M, 2 * np.abs(M).sum(1))
    d = 1 / np.sqrt(np.diagonal(M))
    return d[:, None] * M * d[None, :]


@pytest.mark.parametrize("s", [0, 20, 30, 40, 100])
@pytest.mark.parametrize("n, leaf, col", [(128, 64, 63), (128, 64, 20), (256, 128, 127), (300, 64, 10)])
def test_a_row_of_other_units_keeps_its_neighbours_in_a_factor(env, n, leaf, col, s):
    """A = D M D, the column in units 2^-s; one row of the panel below couples to that column alone."""
    hrp, h, _ = env
    rng = np.random.default_rng(n + col)
    A = _dominant(n, rng)
    row = leaf + 5
    A[row, :row] = A[:row, row] = 0.0
    A[row, col] = A[col, row] = 0.3
    d = np.ones(n)
    d[col] = 2.0 ** -s
    A = d[:, None] * A * d[None, :]
    At = hrp.colmajor(A).cuda()
    assert h.potrf(hrp.tree_parse("[F64]", leaf=leaf), At) == 0
    L = np.tril(hrp.from_colmajor(At)).astype(np.longdouble)
    err = np.abs(A - L @ L.T)
    sd = np.sqrt(np.diagonal(A))
    assert np.all(err <= 4 * (n + 1) * 2.0 ** -53 * np.outer(sd, sd)), float(np.max(err / np.outer(sd, sd)))


@pytest.mark.parametrize("kind", ["entries", "one column", "one row", "identity"])
@pytest.mark.parametrize("m, n, s", [(130, 57, 20), (133, 64, 40), (200, 100, 40), (2500, 128, 20), (2433, 64, 60)])
def test_entries_are_accurate_against_their_own_terms(env, m, n, s, kind):
    hrp, h, _ = env
    rng = np.random.default_rng(m + n)
    L = np.tril(rng.standard_normal((n, n))) / (4 * n)
    L[np.arange(n), np.arange(n)] = 1 + rng.random(n)
    X = rng.standard_normal((m, n))
    if kind == "entries":
        X *= np.exp2(rng.integers(-s, s, (m, n)))
    elif kind == "one column":                                 # large in every seventh row
        X[::7, n // 3] *= 2.0 ** s
    elif kind == "one row":
        X[m // 2] *= np.exp2(rng.integers(-s, s, n))
    B = X @ L.T if kind != "identity" else np.eye(m, n)
    Bt = hrp.colmajor(B).cuda()
    h.trsm(hrp.tree_parse("[F64]", leaf=128), hrp.colmajor(L).cuda(), Bt)
    assert h.check() == 0
    Xq, Lq = hrp.from_colmajor(Bt).astype(np.longdouble), L.astype(np.longdouble)
    rows = slice(None) if m < 1000 else slice(m - 140, m)
    res = np.abs(B[rows] - Xq[rows] @ Lq.T)
    bound = 4 * n * np.longdouble(2.0) ** -53 * (np.abs(Xq[rows]) @ np.abs(Lq).T)
    assert np.all(res <= bound), float(np.max(res / np.where(bound > 0, bound, 1)))
    if kind == "identity":
        assert np.all(np.triu(Xq[:n].T, 1) == 0)
