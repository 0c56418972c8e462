"""The refinement's residual by digit products, seen through hrp_posv with max_iter = 0 on the
FP64 tree: the reported residual must be that of the returned X, and GMRES products (the same
kernel) must converge.  Orders at block edges (64), every right-hand-side grouping (8, 16, a second
pass), matrices scaled over many decades, and an indefinite matrix (the FP64 FMA path)."""
import numpy as np
import pytest

from synth import dominant_spd, rhs, seed_for, wide_range_spd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    yield hrp, h, torch
    h.close()


def _posv(env, A, B, tree, max_iter):
    hrp, h, torch = env
    At, Bt = hrp.colmajor(A).cuda(), hrp.colmajor(B).cuda()
    X = torch.zeros_like(Bt)
    r = h.posv(hrp.tree_parse(tree, leaf=128), At, Bt, X, max_iter=max_iter, tol=1e-15)
    return r, hrp.from_colmajor(X)


def _check(A, B, X, resid):
    """The reported residual against extended precision: FP64 evaluation of b - A x may add
    at most (n + 2) 2^-53 |A||x| per entry."""
    n = A.shape[0]
    r = B.astype(np.longdouble) - A.astype(np.longdouble) @ X.astype(np.longdouble)
    slack = (n + 2) * 2.0 ** -53 * (np.abs(A) @ np.abs(X) + np.abs(B))
    nb = np.linalg.norm(B, axis=0)
    true = float((np.linalg.norm(r.astype(float), axis=0) / nb).max())
    dev = float((np.linalg.norm(slack, axis=0) / nb).max())
    assert abs(resid - true) <= dev, (resid, true, dev)


@pytest.mark.parametrize("n,nrhs", [(1, 1), (63, 1), (64, 8), (65, 9), (129, 16), (300, 17), (777, 3)])
def test_reported_residual_is_the_true_one(env, n, nrhs):
    A = dominant_spd(n, 2.0, seed_for(21, n)) if n > 1 else np.array([[3.0]])
    B = rhs(n, nrhs, seed_for(22, n))
    r, X = _posv(env, A, B, "[F32|F64@128]", 0)
    assert r["info"] == 0
    _check(A, B, X, r["resid"])


def test_residual_of_a_matrix_over_many_decades(env):
    A = wide_range_spd(200, 24, seed_for(23, 1))
    B = A @ rhs(200, 2, seed_for(23, 2))
    r, X = _posv(env, A, B, "[F64]", 0)
    assert r["info"] == 0
    _check(A, B, X, r["resid"])
