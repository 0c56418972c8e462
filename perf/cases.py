"""The work this library is measured on: factorizations, solves and BLAS-3 calls through the
public Python binding (one call of the C ABI each), over the sizes, trees and options that its
tests, its benchmark and its configurations use.

Matrices are column-major FP64 in row-major torch tensors T of shape (columns, ld), T[j, i] =
M(i, j), as everywhere in the binding.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2601_08082_gb300 as hrp

FP64 = "[F64]"
FALLBACK = "[F32|F64@128]"
SHALLOW = "[F16,F32|F64@128]"
MIDDLE = "[F16,F16,F32|F64@128]"
DEEP = "[F16,F16,F16,F16,F32|F64@128]"
FP8 = "[F8,F16,F16,F32|F64@128]"
PURE16 = "[F16]"

RHOS = (1.05, 2.0, 8.0)
MAX_ITER, TOL = 30, 1e-12


def listed():
    return [
        # The smallest call a program makes: one little FP64 system, all launches and latency.
        dict(name="factor_solve_fp64_n96", kind="factor_solve", tree=FP64, leaf=64, n=96, nrhs=1, pad=0, rho=1.05),
        # The plain FP64 recursion of the first configuration: n = 1024, leaf 64, one right-hand side.
        dict(name="factor_solve_fp64_n1024", kind="factor_solve", tree=FP64, leaf=64, n=1024, nrhs=1, pad=0, rho=1.05),
        # An ordinary solve to FP64 accuracy on a mixed tree: an order that divides by nothing, a
        # padded leading dimension, a few right-hand sides.
        dict(name="posv_mixed_n1999_r3", kind="posv", tree=SHALLOW, leaf=128, n=1999, nrhs=3, pad=4, rho=2.0),
        # The benchmark's headline step: n = 8192, FP16 outer levels, one right-hand side.
        dict(name="factor_solve_mixed_n8192", kind="factor_solve", tree=DEEP, leaf=128, n=8192, nrhs=1, pad=0, rho=2.0),
        # A factor kept from before, applied to new right-hand sides (time stepping, sampling).
        dict(name="solve_n4096_r16", kind="solve", tree=FP64, leaf=128, n=4096, nrhs=16, pad=0, rho=2.0),
        # The same on the conservative tree, one right-hand side, a barely dominant matrix.
        dict(name="posv_fallback_n2500", kind="posv", tree=FALLBACK, leaf=128, n=2500, nrhs=1, pad=0, rho=1.05),
        # A block of right-hand sides on a deeper mixed tree.
        dict(name="posv_mixed_n4096_r16", kind="posv", tree=MIDDLE, leaf=128, n=4096, nrhs=16, pad=0, rho=2.0),
        # The largest configuration: n = 32768, FP8 outermost level, 16 right-hand sides.
        dict(name="posv_fp8_n32768_r16", kind="posv", tree=FP8, leaf=128, n=32768, nrhs=16, pad=0, rho=2.0),
        # Many systems of uneven orders in one call, refined to FP64 accuracy.
        dict(name="batched_posv_48", kind="batched_posv", tree=SHALLOW, leaf=128, batch=48, lo=64, hi=2048, nrhs=4,
             sizes=1),
        # Many kernel matrices (Gaussian-process fits) factored and solved in FP64.
        dict(name="batched_fp64_rbf_24", kind="batched_fp64", tree=FP64, leaf=64, batch=24, lo=64, hi=1024, nrhs=4,
             sizes=2),
        # The standalone recursive kernels of the paper's SYRK and TRSM experiments.
        dict(name="syrk_mixed_n4000_k1024", kind="syrk", tree=MIDDLE, leaf=128, n=4000, k=1024),
        dict(name="trsm_mixed_m3000_n2048", kind="trsm", tree=MIDDLE, leaf=128, m=3000, n=2048, rho=2.0),
    ]


def _order(rng, lo, hi):
    """An order drawn uniformly in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["factor_solve", "factor_solve", "factor_solve", "solve", "posv", "posv", "batched_posv",
                       "batched_fp64", "syrk", "trsm"])
    rho = rng.choice(RHOS)
    if kind == "factor_solve":
        # FP64 factors over the small and middle orders, mixed ones over the large orders (smaller
        # mixed systems are solved through posv, which refines them)
        fp64 = rng.random() < 0.6
        n = _order(rng, 64, 2048) if fp64 else _order(rng, 8192, 16384)
        return dict(kind=kind, tree=FP64 if fp64 else rng.choice([MIDDLE, DEEP]), leaf=64 if fp64 else 128, n=n,
                    nrhs=rng.choice([1, 1, 3, 16]), pad=rng.choice([0, 0, 1, 8]), rho=rho if fp64 else max(rho, 2.0))
    if kind == "solve":
        return dict(kind=kind, tree=FP64, leaf=128, n=_order(rng, 64, 8192), nrhs=rng.choice([1, 2, 4, 7, 16, 20]),
                    pad=rng.choice([0, 0, 3]), rho=rho)
    if kind == "posv":
        tree = rng.choice([FALLBACK, SHALLOW, MIDDLE, DEEP, FP8])
        n = 128 * 2 ** rng.randint(4, 7) if tree == FP8 else _order(rng, 128, 8192)
        return dict(kind=kind, tree=tree, leaf=128, n=n, nrhs=rng.choice([1, 2, 4, 16]), pad=rng.choice([0, 0, 2]),
                    rho=rho)
    if kind in ("batched_posv", "batched_fp64"):
        posv = kind == "batched_posv"
        return dict(kind=kind, tree=SHALLOW if posv else FP64, leaf=128 if posv else 64, batch=rng.randint(4, 40),
                    lo=64, hi=rng.choice([256, 512, 1024]), nrhs=rng.choice([1, 2, 4]), sizes=rng.randrange(1 << 20))
    tree = rng.choice([FP64, FALLBACK, MIDDLE, PURE16]) if kind == "syrk" else rng.choice([FP64, FALLBACK, MIDDLE])
    top = 2048 if tree == FP64 else 4096
    if kind == "syrk":
        return dict(kind=kind, tree=tree, leaf=128, n=_order(rng, 128, top), k=_order(rng, 64, 2048))
    return dict(kind=kind, tree=tree, leaf=128, m=_order(rng, 128, top), n=_order(rng, 128, 2048), rho=rho)


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _dominant(g, n, rho):
    """(B + B^T) / 2 with B iid N(0, 1) and a_ii = rho sum_{j != i} |a_ij|."""
    B = _randn(g, n, n)
    A = B + B.T
    del B
    A.mul_(0.5)
    d = A.diagonal()
    d.zero_()
    s = torch.linalg.vector_norm(A, ord=1, dim=1)
    A.diagonal().copy_(s.mul_(rho).clamp_(min=1.0))
    return A


def _rbf(g, n):
    """exp(-|x_i - x_j|^2 / (2 0.5^2)) of points in the unit cube, plus 1e-2 on the diagonal."""
    x = torch.rand(n, 3, dtype=torch.float64, device="cuda", generator=g)
    A = torch.exp(-2.0 * (x[:, None, :] - x[None, :, :]).square().sum(-1))
    A.diagonal().add_(1e-2)
    return A


def _padded(A, pad):
    """The column-major buffer of the symmetric A with `pad` unused rows under each column."""
    if not pad:
        return A
    out = torch.zeros(A.shape[0], A.shape[1] + pad, dtype=A.dtype, device=A.device)
    out[:, :A.shape[1]] = A
    return out


def _buffers(shapes):
    """Zeroed results of many systems in one allocation: the flat buffer and its
    views of the given shapes, each starting on a 256-byte boundary."""
    starts, at = [], 0
    for a, b in shapes:
        starts.append(at)
        at += (a * b + 31) // 32 * 32
    flat = torch.zeros(at, dtype=torch.float64, device="cuda")
    return flat, [flat[o:o + a * b].view(a, b) for o, (a, b) in zip(starts, shapes)]


def _flattened(arrays):
    flat, views = _buffers([tuple(a.shape) for a in arrays])
    for v, a in zip(views, arrays):
        v.copy_(a)
    return flat


def _orders(case):
    r = random.Random(case["sizes"])
    return [r.randint(case["lo"], case["hi"]) for _ in range(case["batch"])]


def _inputs(case, seed):
    """The arrays of a case, from the seed alone (exact() draws the same ones)."""
    g, kind = _gen(seed), case["kind"]
    if kind in ("factor_solve", "solve", "posv"):
        A = _dominant(g, case["n"], case["rho"])
        return {"A": A, "B": _randn(g, case["nrhs"], case["n"])}
    if kind == "batched_posv":
        ns = _orders(case)
        return {"A": [_dominant(g, n, RHOS[i % 3]) for i, n in enumerate(ns)], "B": [_randn(g, case["nrhs"], n) for n in ns]}
    if kind == "batched_fp64":
        ns = _orders(case)
        return {"A": [_rbf(g, n) for n in ns], "B": [_randn(g, case["nrhs"], n) for n in ns]}
    if kind == "syrk":
        n, k = case["n"], case["k"]
        A = _randn(g, k, n)                              # column-major n x k
        C = _randn(g, n, n)
        return {"A": A, "C": C + C.T}
    m, n = case["m"], case["n"]
    # a factor's triangle, scaled as the factor of a dominant matrix is
    L = _randn(g, n, n)
    L.mul_(1.0 / math.sqrt(n))
    L.diagonal().abs_().add_(case["rho"] * math.sqrt(n))
    return {"L": L, "B": _randn(g, n, m)}                # B column-major m x n


def prepare(case, seed):
    """A program's matrices and right-hand sides on the GPU, its buffers for the results, the
    parsed tree and its handle; for `solve`, also the factor it kept."""
    x = _inputs(case, seed)
    st = {"kind": case["kind"], "h": hrp.Handle(torch.cuda.current_device()),
          "tree": hrp.tree_parse(case["tree"], leaf=case["leaf"])}
    kind = case["kind"]
    if kind in ("factor_solve", "solve", "posv"):
        st["A"], st["B"] = _padded(x["A"], case["pad"]), x["B"]
        st["X"] = torch.empty_like(x["B"])
        if kind != "posv":
            st["info"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        if kind == "factor_solve":
            st["L"] = torch.empty_like(st["A"])
        if kind == "solve":
            st["h"].potrf_async(st["tree"], st["A"], st["info"])
    elif kind in ("batched_posv", "batched_fp64"):
        st["A"], st["B"] = x["A"], x["B"]
        st["Xflat"], st["X"] = _buffers([tuple(b.shape) for b in x["B"]])
        if kind == "batched_fp64":
            st["Lflat"], st["L"] = _buffers([tuple(a.shape) for a in x["A"]])
            st["info"] = torch.zeros(case["batch"], dtype=torch.int32, device="cuda")
    elif kind == "syrk":
        st["A"], st["C"], st["out"] = x["A"], x["C"], torch.empty_like(x["C"])
    else:
        st["L"], st["B"], st["out"] = x["L"], x["B"], torch.empty_like(x["B"])
    return st


def run(st):
    """One pass.  The calls that work in place take a copy, so that the inputs last."""
    h, tree, kind = st["h"], st["tree"], st["kind"]
    if kind == "factor_solve":
        st["L"].copy_(st["A"])
        st["X"].copy_(st["B"])
        h.potrf_async(tree, st["L"], st["info"])
        h.potrs(st["L"], st["X"])
        return {"L": st["L"], "X": st["X"], "info": st["info"]}
    if kind == "solve":
        st["X"].copy_(st["B"])
        h.potrs(st["A"], st["X"])
        return {"X": st["X"]}
    if kind == "posv":
        r = h.posv(tree, st["A"], st["B"], st["X"], max_iter=MAX_ITER, tol=TOL)
        return {"X": st["X"], "status": r["status"], "info": r["info"], "used_fallback": r["used_fallback"]}
    if kind == "batched_posv":
        r = h.posv_batched(tree, st["A"], st["B"], st["X"], max_iter=MAX_ITER, tol=TOL)
        return {"X": st["Xflat"], "status": r["status"], "info": np.array(r["info"], dtype=np.int32)}
    if kind == "batched_fp64":
        torch._foreach_copy_(st["L"], st["A"])
        torch._foreach_copy_(st["X"], st["B"])
        h.potrf_batched(tree, st["L"], st["info"])
        h.potrs_batched(st["L"], st["X"])
        return {"L": st["Lflat"], "X": st["Xflat"], "info": st["info"]}
    st["out"].copy_(st["C"] if kind == "syrk" else st["B"])
    if kind == "syrk":
        h.syrk(tree, st["A"], st["out"])
    else:
        h.trsm(tree, st["L"], st["out"])
    return {"out": st["out"]}


# ---------------------------------------------------------------------------------------
# What a pass cannot do without, and what it should return
# ---------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    tri = lambda n: n * (n + 1) // 2
    if kind == "factor_solve":
        n, r = case["n"], case["nrhs"]
        return {"bytes": 8 * (2 * tri(n) + 2 * n * r), "flops": n ** 3 / 3 + 2.0 * n * n * r}
    if kind == "solve":
        n, r = case["n"], case["nrhs"]
        return {"bytes": 8 * (tri(n) + 2 * n * r), "flops": 2.0 * n * n * r}
    if kind == "posv":
        n, r = case["n"], case["nrhs"]
        return {"bytes": 8 * (tri(n) + 2 * n * r), "flops": n ** 3 / 3 + 2.0 * n * n * r}
    if kind in ("batched_posv", "batched_fp64"):
        ns, r, w = _orders(case), case["nrhs"], 1 if kind == "batched_posv" else 2
        return {"bytes": 8 * sum(w * tri(n) + 2 * n * r for n in ns),
                "flops": sum(n ** 3 / 3 + 2.0 * n * n * r for n in ns)}
    if kind == "syrk":
        n, k = case["n"], case["k"]
        return {"bytes": 8 * (n * k + 2 * tri(n)), "flops": 1.0 * n * (n + 1) * k}
    m, n = case["m"], case["n"]
    return {"bytes": 8 * (tri(n) + 2 * m * n), "flops": 1.0 * m * n * n}


def _solve64(A, B):
    """A^{-1} B^T as rows, in FP64: by Cholesky, or by conjugate gradients (dominant matrices,
    run to the last bits) where a Cholesky factorization would take many seconds."""
    if A.shape[0] <= 16384:
        return torch.cholesky_solve(B.T.contiguous(), torch.linalg.cholesky(A)).T.contiguous()
    X = torch.zeros_like(B)
    R, P = B.clone(), B.clone()
    rr = (R * R).sum(1, keepdim=True)
    for _ in range(60):
        Q = P @ A
        a = rr / (P * Q).sum(1, keepdim=True)
        X += a * P
        R -= a * Q
        new = (R * R).sum(1, keepdim=True)
        P = R + (new / rr) * P
        rr = new
        if float((rr.sqrt() / B.norm(dim=1, keepdim=True)).max()) < 1e-17:
            break
    return X


def _factored(A, pad):
    """The buffer after a factorization: L in the matrix's lower triangle (the storage's upper
    one), the rest as it was."""
    L = torch.linalg.cholesky(A)
    out = torch.triu(L.T) + torch.tril(A, -1)
    return _padded(out, pad)


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "factor_solve":
        return {"L": _factored(x["A"], case["pad"]), "X": _solve64(x["A"], x["B"]), "info": None}
    if kind == "solve":
        return {"X": _solve64(x["A"], x["B"])}
    if kind == "posv":
        return {"X": _solve64(x["A"], x["B"]), "status": None, "info": None, "used_fallback": None}
    if kind == "batched_posv":
        return {"X": _flattened([_solve64(a, b) for a, b in zip(x["A"], x["B"])]), "status": None, "info": None}
    if kind == "batched_fp64":
        return {"L": _flattened([_factored(a, 0) for a in x["A"]]),
                "X": _flattened([_solve64(a, b) for a, b in zip(x["A"], x["B"])]), "info": None}
    if kind == "syrk":
        full = x["C"] - x["A"].T @ x["A"]
        return {"out": torch.triu(full) + torch.tril(x["C"], -1)}
    # X L^T = B with column-major storage: the stored rows solve L Y = B
    L = torch.tril(x["L"].T)
    return {"out": torch.linalg.solve_triangular(L, x["B"], upper=False)}
