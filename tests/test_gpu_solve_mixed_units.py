"""Solves with factors whose rows are in different units: the block inverses of hrp_potrs, one right-hand
side, against the residual of L L^T x = b entry by entry.

Bound: with a block's inverse W the solution of L y = b is y = W b up to 2 n 2^-53 |W| |b| (W itself
within n 2^-53 |W| |L| |W|, the product's roundings), so the residual is at most 2 n 2^-53 |L| |W| |b| <=
2 n 2^-53 |L| |W| |L| |y|, and the same again for the transpose.  The doubling's products hold an
output to 2^-59.7 of scales that are at most 2^14 times its terms: n 2^-45.7 in place of n 2^-53 for the
few outputs near that line, which 2^4 covers for ordinary digits.
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


def _factor(n, rng):
    """The factor of a dominant matrix with unit diagonal: |W| |L| stays small."""
    B = rng.standard_normal((n, n))
    A = (B + B.T) / 2
    np.fill_diagonal(A, 0)
    np.fill_diagonal(A, 2 * np.maximum(np.abs(A).sum(1), 1))
    d = 1 / np.sqrt(np.diagonal(A))
    return np.linalg.cholesky(d[:, None] * A * d[None, :])


def _check(L, B, X):
    n = len(L)
    aL, W = np.abs(L), np.abs(np.linalg.inv(L))
    Lq = L.astype(np.longdouble)
    res = np.abs(B - Lq @ (Lq.T @ X.astype(np.longdouble))).astype(float)
    bound = 16 * 4 * n * 2.0 ** -53 * (aL @ (W @ (aL @ (aL.T @ (W.T @ (aL.T @ np.abs(X)))))))
    assert np.all(res <= bound), float(np.max(res / bound))


def _potrs(env, L, B):
    hrp, h, _ = env
    Xt = hrp.colmajor(B).cuda()
    h.potrs(hrp.colmajor(L).cuda(), Xt)
    return hrp.from_colmajor(Xt)


@pytest.mark.parametrize("s", [0, 10, 20, 30, 40, 200])
@pytest.mark.parametrize("n, row, col", [(128, 70, 63), (128, 127, 63), (300, 200, 127), (512, 300, 255), (1300, 400, 255)])
def test_a_row_in_other_units_keeps_its_neighbours(env, n, row, col, s):
    rng = np.random.default_rng(n + row)
    L = _factor(n, rng)
    L[row, :row] = 0.0
    L[row, col] = 0.7
    L[row] *= 2.0 ** s
    b = rng.standard_normal((n, 1))
    b[row] *= 2.0 ** s
    _check(L, b, _potrs(env, L, b))
