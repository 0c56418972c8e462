"""Entries of an FP64 leaf's factor far below their row's and column's scales (weakly coupled unknowns,
banded and sparse matrices): as accurate as an FP64 factorization leaves them, and exact zeros.

Bound: |A - L L^T| <= (n + 1) 2^-53 |L| |L|^T entry by entry (Higham, Thm. 10.3); 4 times that.  It holds
for the entries that are computed again in FP64 and for leaves that are factored directly.
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


def _factor(env, A, leaf=128, chain=None):
    hrp, h, _ = env
    At = hrp.colmajor(A).cuda()
    if chain is not None:
        h.set_leaf_chain(chain)
    try:
        assert h.potrf(hrp.tree_parse("[F64]", leaf=leaf), At) == 0
    finally:
        h.set_leaf_chain(-1)
    return np.tril(hrp.from_colmajor(At))


def _ratio(A, L):
    n = len(A)
    Lq = L.astype(np.longdouble)
    err = np.tril(np.abs(A - Lq @ Lq.T))
    bound = 4 * (n + 1) * np.longdouble(2.0) ** -53 * (np.abs(Lq) @ np.abs(Lq).T)
    return err, bound


@pytest.mark.parametrize("bits", [30, 40, 70, 200])
@pytest.mark.parametrize("n", [9, 33, 64, 100, 128])
def test_weakly_coupled_unknowns(env, n, bits):
    rng = np.random.default_rng(n)
    M = _dominant(n, rng)
    A = np.eye(n) + 2.0 ** -bits * (M - np.eye(n))
    err, bound = _ratio(A, _factor(env, A))
    assert np.all(err <= bound)


@pytest.mark.parametrize("count", [1, 3, 8])
@pytest.mark.parametrize("n", [17, 64, 111, 128])
def test_a_few_small_entries_are_computed_again(env, n, count):
    """Two groups of unknowns, each well coupled inside; `count` unknowns alone, tied to the first by 2^-60."""
    rng = np.random.default_rng(n + count)
    A = _dominant(n, rng)
    alone = rng.choice(np.arange(1, n), count, replace=False)
    A[alone] = 0.0
    A[:, alone] = 0.0
    A[alone, alone] = 1.0
    L0 = _factor(env, A)
    off = ~np.eye(n, dtype=bool)
    assert np.all(L0[alone][:, :][off[alone]] == 0) and np.all(L0[:, alone][off[:, alone]] == 0)      # zeros stay zeros
    A[alone, 0] = A[0, alone] = 2.0 ** -60
    L = _factor(env, A)
    err, bound = _ratio(A, L)
    assert np.all(err[alone] <= bound[alone]), float(np.max(err[alone] / np.where(bound[alone] > 0, bound[alone], 1)))


@pytest.mark.parametrize("n", [64, 128])
def test_small_entries_without_zeros(env, n):
    """Every entry present, four of them tiny: computed again from the refined ones."""
    rng = np.random.default_rng(n)
    A = _dominant(n, rng)
    A[5, 0] = A[0, 5] = 2.0 ** -50
    A[n - 1, 0] = A[0, n - 1] = 2.0 ** -45
    A[n // 2, 0] = A[0, n // 2] = -2.0 ** -70
    L = _factor(env, A)
    for i, v in ((5, 2.0 ** -50), (n - 1, 2.0 ** -45), (n // 2, -2.0 ** -70)):
        assert L[i, 0] == v / L[0, 0]
    err, _ = _ratio(A, L)
    assert np.all(err <= 2.0 ** -51)


@pytest.mark.parametrize("n, band", [(64, 1), (128, 1), (100, 5)])
def test_banded_factors_stay_banded(env, n, band):
    A = np.zeros((n, n))
    for k in range(1, band + 1):
        A += np.diag(np.full(n - k, -1.0 / k), k) + np.diag(np.full(n - k, -1.0 / k), -k)
    A += np.diag(np.abs(A).sum(1) + 0.5)
    L = _factor(env, A)
    assert np.all(np.tril(L, -band - 1) == 0)
    err, bound = _ratio(A, L)
    assert np.all(err <= bound + 2.0 ** -51 * np.abs(A))


def test_direct_and_refined_leaves_agree_on_short_ranged_kernels(env):
    rng = np.random.default_rng(3)
    x = rng.random((100, 3))
    A = np.exp(-200 * ((x[:, None] - x[None]) ** 2).sum(-1)) + 1e-2 * np.eye(100)
    err, bound = _ratio(A, _factor(env, A))
    assert np.all(err <= bound)
