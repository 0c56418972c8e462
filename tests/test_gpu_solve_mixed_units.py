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


# ---- right-hand sides in different units: each column is solved as if it were alone ----
def _check_gpu(torch, L, B, X):
    """_check on the GPU, per column; the residual's own FP64 evaluation adds 4 n 2^-53 |L| |L|^T |x|."""
    n = len(L)
    aL = L.abs()
    W = torch.linalg.solve_triangular(L, torch.eye(n, dtype=L.dtype, device=L.device), upper=False).abs()
    res = (B - L @ (L.T @ X)).abs()
    bound = 68 * n * 2.0 ** -53 * (aL @ (W @ (aL @ (aL.T @ (W.T @ (aL.T @ X.abs()))))))
    assert bool((res <= bound).all()), float((res / bound).max())


def _system(env, n, r):
    _, _, torch = env
    rng = np.random.default_rng(10 * n + r)
    L = torch.from_numpy(_factor(n, rng)).cuda() if n <= 600 else None
    if L is None:
        g = torch.Generator(device="cuda")
        g.manual_seed(n)
        A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
        A = (A + A.T) / 2
        A.diagonal().zero_()
        A.diagonal().copy_(2 * A.abs().sum(1))
        d = torch.rsqrt(A.diagonal())
        L = torch.linalg.cholesky(d[:, None] * A * d[None, :])
    return torch.tril(L), torch.from_numpy(rng.standard_normal((n, r))).cuda()


def _potrs_gpu(env, L, B, pad=0):
    _, h, torch = env
    n, r = B.shape
    Lt = torch.zeros(n, n + pad, dtype=torch.float64, device="cuda")
    Lt[:, :n] = L.T
    Xt = torch.zeros(r, n + pad, dtype=torch.float64, device="cuda")
    Xt[:, :n] = B.T
    h.potrs(Lt, Xt)
    return Xt[:, :n].T


@pytest.mark.parametrize("kind", ["ordinary", "unit", "row", "column"])
@pytest.mark.parametrize("n, r, pad", [(64, 2, 0), (300, 5, 1), (512, 16, 0), (700, 9, 3), (1300, 3, 0), (2500, 2, 1), (2500, 16, 0),
                                       (3001, 9, 3), (4097, 3, 0), (4097, 16, 1)])
@pytest.mark.parametrize("p", [20, 60])
def test_columns_in_other_units_keep_their_neighbours(env, n, r, pad, kind, p):
    _, _, torch = env
    L, B = _system(env, n, r)
    if kind == "unit":                                         # the first column 2^p e_1
        B[:, 0] = 0.0
        B[0, 0] = 2.0 ** p
    elif kind == "row":                                        # all its rows but one in larger units
        B[:, 0] *= 2.0 ** p
        B[n // 2, 0] = 1.0
    elif kind == "column":                                     # all columns apart by 2^p
        B *= torch.exp2(p * torch.arange(r, device="cuda", dtype=torch.float64))[None, :]
    _check_gpu(torch, L, B, _potrs_gpu(env, L, B, pad))


@pytest.mark.parametrize("n", [96, 2500])
def test_unit_vectors(env, n):
    _, _, torch = env
    L, _ = _system(env, n, 1)
    B = torch.eye(n, dtype=torch.float64, device="cuda")[:, n // 3:n // 3 + 16].clone()
    _check_gpu(torch, L, B, _potrs_gpu(env, L, B))


@pytest.mark.parametrize("r", [3, 16])
def test_wide_steps_keep_a_nan_in_its_column(env, r):
    _, _, torch = env
    n = 2500
    L, B = _system(env, n, r)
    B[n // 2, 1] = float("nan")
    X = _potrs_gpu(env, L, B)
    assert bool(torch.isnan(X[:n // 2 + 1, 1]).all())
    keep = [c for c in range(r) if c != 1]
    _check_gpu(torch, L, B[:, keep], X[:, keep])


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_wide_steps_carry_a_bad_entry_of_the_factor(env, bad):
    _, _, torch = env
    n, r = 2500, 3
    L, B = _system(env, n, r)
    L[1800, 30] = bad
    assert bool(torch.isnan(_potrs_gpu(env, L, B)[:1801]).all())


def test_operands_whose_digits_are_all_at_their_lowest(env):
    _, _, torch = env
    a = float(0x207F7F7F7F7F8000) * 2.0 ** -62                 # first digit 33, the others -128
    L = torch.eye(2, dtype=torch.float64, device="cuda")
    L[1, 0] = a
    B = torch.tensor([[a, a], [0.0, 0.0]], dtype=torch.float64, device="cuda")
    X = _potrs_gpu(env, L, B)
    exact = np.longdouble(a) * np.longdouble(a)
    assert abs(np.longdouble(float(X[1, 0])) + exact) <= 2.0 ** -52 * exact
