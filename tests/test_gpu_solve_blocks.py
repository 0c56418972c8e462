"""POTRS by block inverses (orders up to 512 or above 1024, or more than 8 right-hand sides): edges of the
64-, 128-, 256- and 512-row blocks and of the groups of 8 and 16 right-hand sides, ragged leading
dimensions, rows scaled by powers of two from 2^-60 to 2^60, and a NaN in one right-hand side.

Bound: substitution in FP64 solves (L + dL)(L + dL)^T x = b with |dL| <= n 2^-53 |L| (Higham, Thm. 8.5), so
|x - x*| <= 2 n 2^-53 cond(A) |x*| to first order in the norm; the matrices have a_ii = 2 sum_j |a_ij|, whose
condition number after diagonal scaling is at most (1 + 1/2) / (1 - 1/2) = 3; 8 n 2^-53 covers the product.
"""
import pytest

pytestmark = pytest.mark.gpu

CASES = [(n, r) for n in (1, 63, 64, 65, 127, 128, 256, 257, 512) for r in (1, 8)]
CASES += [(n, r) for n in (129, 255, 257, 512, 513, 1024) for r in (9, 17)]
CASES += [(n, r) for n in (1025, 1537) for r in (1, 3, 16)] + [(4096, 3), (4096, 16)]


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    yield h, torch
    h.close()


def _system(torch, n, r):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000 * n + r)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = (A + A.T) / 2
    A.diagonal().zero_()
    A.diagonal().copy_(2 * A.abs().sum(1).clamp_(min=1.0))
    d = torch.rsqrt(A.diagonal())
    A = d[:, None] * A * d[None, :]
    L = torch.linalg.cholesky(A)
    B = torch.randn(n, r, dtype=torch.float64, device="cuda", generator=g)
    X = torch.cholesky_solve(B, L)
    for _ in range(2):
        X += torch.cholesky_solve(B - L @ (L.T @ X), L)
    e = torch.randint(-60, 61, (n,), device="cuda", generator=g)
    return L, B, X, torch.exp2(e.to(torch.float64))


def _potrs(h, torch, L, B, pad):
    """X by the library, from column-major copies with `pad` unused rows; the rest stays as it was."""
    n, r = B.shape
    Lt = torch.full((n, n + pad), 7.0, dtype=torch.float64, device="cuda")
    Lt[:, :n] = torch.triu(L.T) + torch.tril(torch.full_like(L, float("nan")), -1)     # the upper triangle is not read
    Bt = torch.full((r, n + pad), 5.0, dtype=torch.float64, device="cuda")
    Bt[:, :n] = B.T
    h.potrs(Lt, Bt)
    assert bool((Bt[:, n:] == 5.0).all())
    return Bt[:, :n].T


@pytest.mark.parametrize("scaled", [False, True])
@pytest.mark.parametrize("n, r", CASES)
def test_block_solve_meets_the_substitution_bound(env, n, r, scaled):
    h, torch = env
    L, B, X, d = _system(torch, n, r)
    if scaled:
        out = _potrs(h, torch, d[:, None] * L, d[:, None] * B, 3) * d[:, None]
    else:
        out = _potrs(h, torch, L, B, n % 2)
    err = torch.linalg.vector_norm(out - X, dim=0) / torch.linalg.vector_norm(X, dim=0)
    assert float(err.max()) <= 8 * n * 2.0 ** -53


@pytest.mark.parametrize("n, r", [(100, 8), (700, 16), (1300, 3)])
def test_block_solve_keeps_a_nan_in_its_column(env, n, r):
    h, torch = env
    L, B, X, _ = _system(torch, n, r)
    B[n // 2, 1] = float("nan")
    out = _potrs(h, torch, L, B, 0)
    assert bool(torch.isnan(out[:n // 2 + 1, 1]).all())
    out[:, 1] = X[:, 1]
    err = torch.linalg.vector_norm(out - X, dim=0) / torch.linalg.vector_norm(X, dim=0)
    assert float(err.max()) <= 8 * n * 2.0 ** -53
