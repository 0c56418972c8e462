"""FP64-level products whose operands' columns or entries are in different units (hrp_syrk, and the
updates between the leaves of hrp_trsm, all-FP64 trees): an entry of the result is accurate against its
own terms, not against its rows' largest ones.

Bounds (derived, per entry): a digit product holds every term to 2^-59.7 of the two scales' product and is
used where sum |x| |y| is at least 2^-8 of it, so k 2^-51.7 sum |x| |y|; the product's and the
subtraction's roundings add 2^-52 (|c| + 2 sum |x| |y|).  Substitution leaves a residual of n 2^-53 |X|
|L|^T (Higham, Thm. 8.5), with the updates 4 n 2^-53 in all.
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


def _syrk(env, A, C0):
    hrp, h, _ = env
    Ct = hrp.colmajor(C0).cuda()
    h.syrk(hrp.tree_parse("[F64]", leaf=16), hrp.colmajor(A).cuda(), Ct)
    assert h.check() == 0
    return np.tril(hrp.from_colmajor(Ct))


def test_syrk_keeps_an_entry_made_of_its_rows_small_terms(env):
    out = _syrk(env, np.array([[1.0, 2.0 ** -70], [0.0, 1.0]]), np.zeros((2, 2)))
    assert out[1, 0] == -2.0 ** -70 and out[0, 0] == -1.0 and out[1, 1] == -1.0


@pytest.mark.parametrize("kind", ["entries", "columns", "halves", "few rows"])
@pytest.mark.parametrize("n, k, s", [(33, 5, 40), (70, 64, 20), (70, 64, 40), (65, 300, 200)])
def test_syrk_is_accurate_against_each_entrys_terms(env, n, k, s, kind):
    rng = np.random.default_rng(n + k + s)
    A = rng.standard_normal((n, k))
    if kind == "entries":
        A *= np.exp2(rng.integers(-s, s, (n, k)))
    elif kind == "columns":
        A *= np.exp2(rng.integers(-s, s, k))[None, :]
    elif kind == "halves":                                     # even rows large where odd ones are small
        A *= np.exp2(s * np.where((np.arange(k)[None, :] + np.arange(n)[:, None]) % 2, 1.0, -1.0))
    else:                                                      # three rows with one large term
        A[[1, n // 2, n - 1], k // 2] *= 2.0 ** s
    C0 = np.zeros((n, n))
    out = _syrk(env, A, C0)
    L = A.astype(np.longdouble)
    ref = np.tril(C0.astype(np.longdouble) - L @ L.T)
    mag = np.abs(L) @ np.abs(L).T
    bound = 2.0 ** -52 * (np.abs(C0) + 2 * mag) + k * 2.0 ** -51.7 * mag
    low = np.tril_indices(n)
    assert np.all(np.abs(out - ref)[low] <= bound[low]), float(np.max(np.abs(out - ref)[low] / bound[low]))


def _triangle(n, kind, s, rng):
    if kind == "rbf":                                          # the factor of a kernel matrix with nugget 10^-s
        x = rng.random((n, 3))
        return np.linalg.cholesky(np.exp(-2 * ((x[:, None] - x[None]) ** 2).sum(-1)) + 10.0 ** -s * np.eye(n))
    L = np.tril(rng.standard_normal((n, n))) / np.sqrt(n)
    L[np.arange(n), np.arange(n)] = 2 + rng.random(n)
    return L * np.exp2(rng.integers(-s, s + 1, n))[None, :]


@pytest.mark.parametrize("kind, s", [("columns", 0), ("columns", 10), ("columns", 20), ("columns", 40), ("rbf", 6), ("rbf", 12)])
@pytest.mark.parametrize("m, n, leaf", [(140, 256, 128), (70, 130, 32), (97, 300, 64)])
def test_trsm_of_several_leaves_meets_the_substitution_bound(env, m, n, leaf, kind, s):
    hrp, h, _ = env
    rng = np.random.default_rng(m + n + s)
    L = _triangle(n, kind, s, rng)
    B = rng.standard_normal((m, n))
    Bt = hrp.colmajor(B).cuda()
    h.trsm(hrp.tree_parse("[F64]", leaf=leaf), hrp.colmajor(L).cuda(), Bt)
    assert h.check() == 0
    X, Lq = hrp.from_colmajor(Bt).astype(np.longdouble), L.astype(np.longdouble)
    res = np.abs(B.astype(np.longdouble) - X @ Lq.T)
    bound = 4 * n * np.longdouble(2.0) ** -53 * (np.abs(X) @ np.abs(Lq).T)
    assert np.all(res <= bound), float(np.max(res / bound))
