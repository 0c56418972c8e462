"""FP32-level TRSM nodes in one launch: two to eight leaves, ragged leaves and rows, rows at and past
the line where the separate launches take over, FP16 copies, with and without FP32 copies of L.

The node runs the same FMAs in the same order as the launches it replaces, in the same rounding, so the
factor with an FP32 copy of L (single call), without (batched call) and with the node split over the
lookahead's streams agree to the bit; and FP32 substitution gives |A - L L^T| <= 2 (n + 1) 2^-24 |L| |L|^T
(Higham, Thm. 10.3; the factor 2 for the inverses of the leaves, whose condition number is below 2 here)
with |L| |L|^T <= sqrt(a_ii a_jj) entrywise.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tree", ["[F32]", "[F16,F32|F64@128]"])
@pytest.mark.parametrize("n, leaf", [(257, 128), (300, 128), (511, 128), (640, 40), (777, 64), (1024, 128), (2049, 128),
                                     (2600, 128)])
def test_trsm_node_agrees_with_itself_and_the_bound(tree, n, leaf):
    import torch

    import paper_2601_08082_gb300 as hrp
    h = hrp.Handle(0)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + leaf)
    A = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    A = (A + A.T) / 2
    A.diagonal().zero_()
    A.diagonal().copy_(2 * A.abs().sum(1))
    t = hrp.tree_parse(tree, leaf=leaf)
    one = A.clone()
    assert h.potrf(t, one) == 0
    many = [A.clone(), A.clone()]
    info = torch.ones(2, dtype=torch.int32, device="cuda")
    h.potrf_batched(t, many, info)
    torch.cuda.synchronize()
    assert info.tolist() == [0, 0]
    assert torch.equal(one, many[0]) and torch.equal(one, many[1])
    L = torch.triu(one).T
    d = torch.sqrt(A.diagonal())
    u = 2.0 ** -24 if "F16" not in tree else 2.0 ** -11
    err = (A - L @ L.T).abs() / (d[:, None] * d[None, :])
    assert float(err.max()) <= 2 * (n + 1) * u
    h.close()
