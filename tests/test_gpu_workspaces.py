"""Workspaces that a call can do without: where they cannot be allocated (a refused allocation, a first call
inside a capture) the call takes the path that needs none, reports nothing, and can be captured."""
import numpy as np
import pytest

from oracle import dense
from synth import dominant_spd, rhs, seed_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mod():
    import torch

    import paper_2601_08082_gb300 as hrp
    return hrp, torch


def _factor(hrp, n):
    A = dominant_spd(n, 2.0, seed_for(9, n))
    L, _ = dense.cholesky(A)
    return A, L, hrp.colmajor(L).cuda()


def _close(a, b):
    return np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("n, r", [(100, 1), (700, 9), (1300, 3)])
def test_solve_without_the_inverses_workspace(mod, n, r):
    hrp, torch = mod
    h = hrp.Handle(0)
    h.alloc_selftest(1)
    _, L, Lt = _factor(hrp, n)
    B = rhs(n, r, seed_for(9, r))
    ref = dense.potrs(L, B)
    Bt = hrp.colmajor(B).cuda()
    X = Bt.clone()
    h.potrs(Lt, X)                                             # refused: the sweeps
    assert h._lib.hrp_last_error(h._h) == b""
    assert _close(hrp.from_colmajor(X), ref)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        X.copy_(Bt)
        h.potrs(Lt, X)
    for _ in range(2):
        X.zero_()
        g.replay()
        assert _close(hrp.from_colmajor(X), ref)
    h.alloc_selftest(0)                                        # the device holds it: the block inverses
    Y = Bt.clone()
    h.potrs(Lt, Y)
    assert _close(hrp.from_colmajor(Y), ref)
    assert not torch.equal(X, Y)
    h.close()


def test_a_solve_captured_before_its_inverses_exist(mod):
    """The order's first call took the sweeps (one right-hand side); nine would take the inverses."""
    hrp, torch = mod
    h = hrp.Handle(0)
    n = 700
    _, L, Lt = _factor(hrp, n)
    B = rhs(n, 9, seed_for(9, 1))
    b1 = hrp.colmajor(B[:, :1]).cuda()
    h.potrs(Lt, b1)
    Bt = hrp.colmajor(B).cuda()
    X = torch.zeros_like(Bt)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        X.copy_(Bt)
        h.potrs(Lt, X)
    g.replay()
    assert _close(hrp.from_colmajor(X), dense.potrs(L, B))
    h.close()


def test_posv_without_the_inverses_workspace(mod):
    hrp, torch = mod
    h = hrp.Handle(0)
    h.alloc_selftest(1)
    n = 600
    A = dominant_spd(n, 2.0, seed_for(9, n))
    B = rhs(n, 4, seed_for(9, 2))
    Xt = torch.empty(4, n, dtype=torch.float64, device="cuda")
    r = h.posv(hrp.tree_parse("[F16,F32|F64@128]", leaf=128), hrp.colmajor(A).cuda(), hrp.colmajor(B).cuda(), Xt)
    assert r["info"] == 0
    X = hrp.from_colmajor(Xt)
    assert np.linalg.norm(A @ X - B) <= 1e-11 * np.linalg.norm(B)
    h.close()


def test_fp64_factor_and_trsm_captured_as_a_handles_first_calls(mod):
    hrp, torch = mod
    n, m = 200, 130
    A, L0, Lt = _factor(hrp, n)
    B = rhs(m, n, seed_for(9, 3))
    tree = hrp.tree_parse("[F64]", leaf=64)
    At, Bt = hrp.colmajor(A).cuda(), hrp.colmajor(B).cuda()
    warm = hrp.Handle(0)                                       # the kernels are loaded
    warm.potrf(tree, At.clone())
    warm.trsm(tree, Lt, Bt.clone())
    torch.cuda.synchronize()
    h = hrp.Handle(0)
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    W, X = torch.zeros_like(At), torch.zeros_like(Bt)
    warm2 = hrp.Handle(0)                                      # the direct schedules too
    warm2.alloc_selftest(1)
    warm2.potrf(tree, At.clone())
    warm2.trsm(tree, Lt, Bt.clone())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        W.copy_(At)
        X.copy_(Bt)
        h.potrf_async(tree, W, info)
        h.trsm(tree, Lt, X)
    for _ in range(2):
        W.zero_()
        X.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        assert _close(np.tril(hrp.from_colmajor(W)), L0)
        assert _close(hrp.from_colmajor(X) @ L0.T, B)
    for x in (h, warm, warm2):
        x.close()
