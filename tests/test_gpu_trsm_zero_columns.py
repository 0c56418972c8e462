"""FP64 leaf TRSM whose right-hand side starts with zero columns, for triangles far from unit scale: the
columns of X that are zero must not set the scale of the others.

Bound: substitution gives (L + dL) x = b with |dL| <= n 2^-53 |L| for every row (Higham, Thm. 8.5), so the
residual |B - X L^T| <= n 2^-53 |X| |L|^T entrywise; one more n 2^-53 covers the residual's own rounding
in FP64.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [-300, -40, 0, 40, 300])
@pytest.mark.parametrize("n, zeros", [(64, 1), (100, 40), (128, 64), (128, 127), (128, 128)])
def test_zero_columns_keep_the_accuracy_of_the_rest(n, zeros, scale):
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + zeros)
    L = torch.tril(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)) / n ** 0.5
    L.diagonal().abs_().add_(2.0)
    L *= 2.0 ** scale
    B = torch.randn(40, n, dtype=torch.float64, device="cuda", generator=g)
    B[:, :zeros] = 0.0
    X = B.T.contiguous()
    h.trsm(hrp.tree_parse("[F64]", leaf=128), L.T.contiguous(), X)
    X = X.T
    assert bool((X[:, :zeros] == 0.0).all())
    assert bool(((B - X @ L.T).abs() <= 2 * n * 2.0 ** -53 * (X.abs() @ L.abs().T)).all())
    h.close()
