"""FP64 leaves by refinement (orders above 8): every edge of the 16-row tiles and 32-column blocks, on
matrices the refinement converges for and on ones it hands to the direct schedules (ill-conditioned,
indefinite, NaN, entries above sqrt(a_ii a_jj)).

Bound: Cholesky in FP64 gives |A - L L^T| <= (n + 1) 2^-53 |L| |L|^T / (1 - (n + 1) 2^-53) entrywise
(Higham, Thm. 10.3), and |L| |L|^T <= sqrt(a_ii a_jj); one more 2^-53 covers the second factor.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ORDERS = [9, 16, 17, 31, 32, 33, 48, 63, 64, 65, 96, 97, 127, 128]


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    yield hrp, h, torch
    h.close()


def _matrix(n, kind, rng):
    if kind == "dominant":
        B = rng.standard_normal((n, n))
        A = (B + B.T) / 2
        A[np.arange(n), np.arange(n)] = 1.05 * (np.abs(A).sum(1) - np.abs(np.diag(A))) + 1e-3
        return A
    if kind == "edge":                          # diagonal entries just below powers of four
        A = 0.01 * rng.standard_normal((n, n))
        A = (A + A.T) / 2
        A[np.arange(n), np.arange(n)] = np.nextafter(4.0 ** rng.integers(1, 3, n), 0)
        return A
    G = rng.standard_normal((n, max(1, n // 2)))
    A = G @ G.T / max(1, n // 2) + {"gram": 1e-1, "hard": 1e-4, "ill": 1e-11, "wide": 1e-1}[kind] * np.eye(n)
    if kind == "wide":
        d = np.exp2(rng.integers(-400, 400, n).astype(float))
        A = A * d[:, None] * d[None, :]
    return A


def _potrf(env, A):
    hrp, h, torch = env
    At = hrp.colmajor(A).cuda()
    info = h.potrf(hrp.tree_parse("[F64]", leaf=128), At)
    return info, hrp.from_colmajor(At)


@pytest.mark.parametrize("kind", ["dominant", "edge", "gram", "hard", "ill", "wide"])
@pytest.mark.parametrize("n", ORDERS)
def test_refined_leaf_meets_the_fp64_bound(env, n, kind):
    A = _matrix(n, kind, np.random.default_rng(100 * n + len(kind)))
    info, out = _potrf(env, A)
    assert info == 0
    assert np.array_equal(np.triu(out, 1), np.triu(A, 1))
    L = np.tril(out).astype(np.longdouble)
    d = np.sqrt(np.diag(A).astype(np.longdouble))
    err = np.abs(A - L @ L.T) / np.outer(d, d)
    assert np.max(np.tril(err)) <= (n + 2) * 2.0 ** -53, float(np.max(np.tril(err)) * 2.0 ** 53)


@pytest.mark.parametrize("n,col", [(20, 1), (20, 20), (64, 33), (128, 70), (128, 128)])
def test_indefinite_leaf_reports_its_column(env, n, col):
    rng = np.random.default_rng(n + col)
    A = _matrix(n, "dominant", rng)
    A[col - 1, col - 1] = -1.0
    info, _ = _potrf(env, A)
    assert info == col
    A = _matrix(n, "dominant", rng)
    if col < n:
        A[col, col - 1] = A[col - 1, col] = 10.0 * np.sqrt(A[col, col] * A[col - 1, col - 1])   # above sqrt(a_ii a_jj)
        info, _ = _potrf(env, A)
        assert info == col + 1


def test_nan_in_a_leaf_is_reported(env):
    A = _matrix(100, "dominant", np.random.default_rng(1))
    A[60, 40] = np.nan
    info, _ = _potrf(env, A)
    assert info == 61
