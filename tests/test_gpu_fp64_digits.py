"""The FP64-level GEMM by digit products (through hrp_syrk with an all-FP64 tree) at tile edges,
chunk edges, rows of very different scales and rows whose later terms outgrow the first.

Bound (derived, per entry): two FP64 roundings, of the product and of the subtraction, of at most
2^-53 (|c| + sum |x y|) each (one more where sums were moved to FP64 between scales), plus the
digits' truncation: every term is exact to 2^-60 of the two rows' scales' product, and a scale is
at most 2^3 times the row's largest entry.
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


def _operand(n, k, kind, rng):
    A = rng.standard_normal((n, k))
    if kind == "rows":                       # rows of very different scales
        A *= np.exp2(rng.integers(-300, 300, n))[:, None].astype(float)
    elif kind == "growing":                  # entries grow by 2^4 every 32 terms
        A *= np.exp2(4.0 * (np.arange(k) // 32))[None, :]
    elif kind == "sparse":
        A[rng.random((n, k)) < 0.7] = 0.0
        A[:, : min(k, 40)] = 0.0
    return A


def _syrk(env, A, C0):
    hrp, h, torch = env
    Ct = hrp.colmajor(C0).cuda()
    h.syrk(hrp.tree_parse("[F64]", leaf=16), hrp.colmajor(A).cuda(), Ct)
    assert h.check() == 0
    return np.tril(hrp.from_colmajor(Ct))


@pytest.mark.parametrize("kind", ["plain", "rows", "growing", "sparse"])
@pytest.mark.parametrize("n,k", [(1, 1), (16, 31), (33, 32), (65, 33), (100, 257), (47, 2081)])
def test_digit_products_meet_the_fp64_bound(env, n, k, kind):
    rng = np.random.default_rng(1000 * n + k)
    A = _operand(n, k, kind, rng)
    C0 = rng.standard_normal((n, n))
    out = _syrk(env, A, C0)
    L = A.astype(np.longdouble)
    ref = np.tril(C0.astype(np.longdouble) - L @ L.T)
    mag = np.abs(A) @ np.abs(A).T
    top = np.abs(A).max(1)
    bound = 2.0 ** -52 * (np.abs(C0) + 2 * mag) + k * 2.0 ** -54 * np.outer(top, top)
    assert np.all(np.abs(out - ref) <= np.tril(bound) + (np.triu(np.ones((n, n)), 1))), \
        float(np.max(np.abs(out - ref)[np.tril_indices(n)] / bound[np.tril_indices(n)]))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_digit_products_carry_nan_and_infinity(env, bad):
    rng = np.random.default_rng(5)
    n, k = 70, 50
    A = rng.standard_normal((n, k))
    A[40, 45] = bad
    C0 = rng.standard_normal((n, n))
    out = _syrk(env, A, C0)
    hit = np.tril(np.add.outer(np.arange(n) == 40, np.arange(n) == 40))
    assert not np.isfinite(out[hit]).any()
    ref = np.tril(C0 - np.delete(A, 45, 1) @ np.delete(A, 45, 1).T - np.outer(np.where(np.arange(n) == 40, 0, A[:, 45]),
                                                                              np.where(np.arange(n) == 40, 0, A[:, 45])))
    keep = np.tril(np.ones((n, n), bool)) & ~hit
    assert np.allclose(out[keep], ref[keep], rtol=0, atol=1e-12)
