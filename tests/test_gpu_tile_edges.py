"""The kernels' tile edges through the C ABI: sizes, column counts, leaf sizes and
panel widths at, below and above the tiles, leading dimensions above n, and both
products.  The bounds are rounding-error bounds (elementwise on |A| |X| where the
kernel is one product), computed from the FP64 reference of each case."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import grad as ograd

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"
U64, U32 = 2.0 ** -53, 2.0 ** -24


def block(X, pad, dtype=torch.float64):
    """The column-major block X on the device with leading dimension n + pad."""
    n, c = X.shape
    t = torch.full((c, n + pad), float("nan"), device=DEV, dtype=dtype)
    t[:, :n] = torch.from_numpy(np.ascontiguousarray(X.T)).to(DEV, dtype)
    return t


def result(t, n, pad):
    assert torch.isnan(t[:, n:]).all() or pad == 0  # rows past n are not written
    return t[:, :n].double().cpu().numpy().T


@pytest.mark.parametrize("prec", ["fp64", "a32"])
@pytest.mark.parametrize("n,c", [(1, 1), (2, 9), (15, 5), (16, 8), (17, 16), (33, 31), (65, 32),
                                 (129, 33), (300, 1), (300, 130), (1025, 40), (2047, 3)])
def test_dense_products(prec, n, c):
    rng = np.random.default_rng(100 * n + c)
    A = rng.standard_normal((n, n)).astype(np.float32).astype(np.float64)
    X = rng.standard_normal((n, c))
    X[: n // 3] = 0.0  # rows of zeros, as in a level's test matrix
    At = torch.from_numpy(A).to(DEV, torch.float64 if prec == "fp64" else torch.float32)
    op = hm.hm_dense_operator_create(At, fp64_blocks=prec == "a32", tensor_cores=False)
    for trans in (0, 1):
        M = A.T if trans else A
        Xd, Y = block(X, 3), block(np.full((n, c), np.nan), 5)
        hm.hm_dense_apply(op, trans, Xd, Y)
        torch.cuda.synchronize()
        err = np.abs(result(Y, n, 5) - M @ X)
        # FP64 products and sums in both precisions: one rounding each
        assert np.all(err <= (n + 8) * U64 * (np.abs(M) @ np.abs(X))), (trans, err.max())


@pytest.mark.parametrize("e", [-80, -1, 80])
def test_split_product_scales_with_the_columns(e):
    """The pre-cut of X is in fixed point relative to each column's window maximum:
    a power of two on X is the same power of two on the product, bit for bit (while
    the sums' units stay in FP32's range); zero columns, and entries more than 2^54 below their column's maximum."""
    n, c = 776, 67
    rng = np.random.default_rng(3)
    A = rng.standard_normal((n, n)).astype(np.float32)
    X = rng.standard_normal((n, c))
    X[:, 5] = 0.0
    X[1::2, 7] *= 2.0 ** -60
    X[:, 9] = np.where(np.arange(n) == 500, 1.0, 0.0)
    op = hm.hm_dense_operator_create(torch.from_numpy(A).to(DEV), fp64_blocks=True, tensor_cores=True)
    for trans in (0, 1):
        out = []
        for s in (1.0, 2.0 ** e):
            Y = block(np.full((n, c), np.nan), 0)
            hm.hm_dense_apply(op, trans, block(X * s, 0), Y)
            torch.cuda.synchronize()
            out.append(result(Y, n, 0))
        assert np.array_equal(out[0] * 2.0 ** e, out[1])
        want = (A.astype(np.float64).T if trans else A.astype(np.float64)) @ X
        assert np.all(out[0][:, 5] == 0.0)
        scale = np.maximum(np.sqrt(np.mean(want ** 2, axis=0)), 1e-300)
        assert (np.abs(out[0] - want) / scale).max() < 3e-8  # orders s + t >= 6 are not formed


def dense_of(h, n, dtype):
    out = torch.empty((n, n), device=DEV, dtype=dtype)
    hm.hm_reconstruct_block(h, 0, n, 0, n, out)
    torch.cuda.synchronize()
    return out.double().cpu().numpy().T


@pytest.mark.parametrize("kind,n,m,r", [("hodlr64", 515, 33, 9), ("hodlr64", 1000, 64, 20),
                                        ("hodlr32", 515, 33, 9), ("hbsid", 1030, 65, 24)])
def test_handle_applies_at_column_counts(kind, n, m, r):
    hodlr = kind.startswith("hodlr")
    A = (W.dense_from_factors(W.synthetic_hodlr_factors(n, m, r - 4, seed=n, shift=float(n))) if hodlr
         else W.log_kernel(n).astype(np.float64))
    mixed = kind == "hodlr32"
    dt = torch.float32 if mixed else torch.float64
    At = torch.from_numpy(A).to(DEV, dt)
    op = hm.hm_dense_operator_create(At)
    t = hm.Tree(n, m)
    if hodlr:
        h = hm.hm_compress_hodlr(op, t, k=r - 4, p=4, seed=2, prec=hm.HM_MIXED if mixed else hm.HM_FP64)
    else:
        h = hm.hm_compress_hbs(op, t, tol=1e-6, r=r, seed=2, prec=hm.HM_FP64)
    Ac = dense_of(h, n, dt)
    rng = np.random.default_rng(n + m)
    for c in (1, 2, 7, 8, 9, 16, 17, 33, 64, 65, 129):
        for trans in (0, 1):
            X = rng.standard_normal((n, c)).astype(np.float32).astype(np.float64)
            Xd, Y = block(X, 2, dt), block(np.full((n, c), np.nan), 3, dt)
            hm.hm_apply(h, trans, Xd, Y)
            torch.cuda.synchronize()
            got, want = result(Y, n, 3), (Ac.T if trans else Ac) @ X
            # products of up to 2 log2(n/m) + 2 factors with orthonormal or bounded
            # bases, n terms in all: n u, with room for the levels
            tol = 16 * n * (U32 if mixed else U64)
            assert np.linalg.norm(got - want) <= tol * np.linalg.norm(Ac) * np.linalg.norm(X) / np.sqrt(n), \
                (c, trans)
            if c in (1, 33, 129):  # Y in X's place, and in alternating columns of one buffer
                Xi = block(X, 2, dt)
                hm.hm_apply(h, trans, Xi, Xi)
                both = torch.empty((2 * c, n), device=DEV, dtype=dt)
                both[::2] = Xd[:, :n]
                hm.hm_apply(h, trans, both[::2], both[1::2])
                torch.cuda.synchronize()
                assert torch.equal(Xi[:, :n], Y[:, :n]) and torch.equal(both[1::2], Y[:, :n])


@pytest.mark.parametrize("n,m,r", [(66, 33, 1), (130, 65, 5), (257, 17, 8), (1000, 250, 33),
                                   (515, 129, 64), (600, 80, 40)])
def test_solver_at_odd_leaves_and_ranks(n, m, r):
    """The block inverses (orders from 2 to 250) at sizes that split unevenly."""
    A = W.dense_from_factors(W.synthetic_hodlr_factors(n, m, r, seed=n + r, shift=float(n)))
    op = hm.hm_dense_operator_create(torch.from_numpy(A).to(DEV))
    h = hm.hm_compress_hodlr(op, hm.Tree(n, m), k=r, p=0, seed=2, prec=hm.HM_FP64)
    Ac = dense_of(h, n, torch.float64)
    hm.hm_hodlr_factorize(h)
    rng = np.random.default_rng(r)
    for c in (1, 9, 40):
        B = rng.standard_normal((n, c))
        for trans in (0, 1):
            Bd, X = block(B, 1), block(np.full((n, c), np.nan), 4)
            hm.hm_solve(h, trans, Bd, X)
            torch.cuda.synchronize()
            got, M = result(X, n, 4), Ac.T if trans else Ac
            want = np.linalg.solve(M, B)
            # a backward-stable solve is accurate to about cond(A_c) u; 100x allowed
            tol = 100.0 * np.linalg.cond(Ac) * U64
            assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want), (c, trans)


@pytest.mark.parametrize("n,m,k", [(62, 31, 1), (125, 32, 3), (131, 33, 32), (255, 64, 17), (259, 65, 64),
                                   (2047, 16, 64), (1500, 750, 5), (4096, 256, 32), (5003, 9, 24)])
def test_factored_layer_at_leaf_and_rank_edges(n, m, k):
    """Apply, adjoint and the fused loss gradient in FP32 against FP64, elementwise
    within the rounding bound of the same sums of absolute values."""
    f = W.synthetic_hodlr_factors(n, m, k, seed=n + k, shift=0.0, dtype=np.float32)
    L, t = f["L"], hm.Tree(n, m)
    sizes = [d.shape[0] for d in f["D"]]
    nmax = max(sizes)
    rng = np.random.default_rng(k)
    x, b = (rng.standard_normal(n).astype(np.float32) for _ in range(2))
    U, V = (torch.from_numpy(np.stack([np.ascontiguousarray(f[s][j].T) for j in range(1, L + 1)])).to(DEV)
            for s in "UV")
    Dp = np.zeros((len(sizes), nmax, nmax), np.float32)  # column-major per leaf
    for l, d in enumerate(f["D"]):
        Dp[l, : d.shape[0], : d.shape[0]] = d.T
    D = torch.from_numpy(Dp).to(DEV)
    xd, bd = torch.from_numpy(x).to(DEV), torch.from_numpy(b).to(DEV)
    fa = dict(f, U=[None] + [np.abs(u) for u in f["U"][1:]], V=[None] + [np.abs(v) for v in f["V"][1:]],
              D=[np.abs(d) for d in f["D"]])
    gamma = (n + L * k + nmax) * U32  # terms of the longest chain of sums
    nan = lambda ref: torch.full_like(ref, float("nan"))

    for trans in (0, 1):
        y = nan(xd)
        hm.hm_hodlr_factored_apply(t, k, U, V, D, xd, y, trans)
        torch.cuda.synchronize()
        xi = xd.clone()
        hm.hm_hodlr_factored_apply(t, k, U, V, D, xi, xi, trans)  # y in x's place
        torch.cuda.synchronize()
        for got in (y, xi):
            err = np.abs(got.cpu().numpy() - ograd.apply(f, x, bool(trans)))
            assert np.all(err <= gamma * ograd.apply(fa, np.abs(x), bool(trans))), trans

    want = ograd.gradients(f, x, b)
    bound = ograd.gradients(fa, np.abs(x), -np.abs(b))
    y, r, gx, gU, gV, gD = nan(xd), nan(xd), nan(xd), nan(U), nan(V), nan(D)

    def check(gx, gU, gV, gD):
        # two chains (the residual's and the adjoint's) and the products of both
        g3 = 3 * gamma
        assert np.all(np.abs(gx.cpu().numpy() - want[0]) <= g3 * bound[0])
        for g, w, bd_ in ((gU, want[1], bound[1]), (gV, want[2], bound[2])):
            for j in range(1, L + 1):
                assert np.all(np.abs(g[j - 1].cpu().numpy().T - w[j]) <= g3 * bd_[j]), j
        for l, s in enumerate(sizes):
            G = gD[l].cpu().numpy().T
            assert np.all(np.abs(G[:s, :s] - want[3][l]) <= g3 * bound[3][l])
            assert np.all(G[s:] == 0.0) and np.all(G[:, s:] == 0.0)

    hm.hm_hodlr_factored_loss_grad(t, k, U, V, D, xd, bd, 2.0, y, r, gx, gU, gV, gD)
    torch.cuda.synchronize()
    check(gx, gU, gV, gD)
    gx2, gU2, gV2, gD2 = nan(xd), nan(U), nan(V), nan(D)
    hm.hm_hodlr_factored_adjoint(t, k, U, V, D, xd, r, 2.0, gx2, gU2, gV2, gD2)
    torch.cuda.synchronize()
    check(gx2, gU2, gV2, gD2)
    for src in (0, 1):  # gx in x's or r's place, gD in D's
        v, Di = [xd.clone(), r.clone()], D.clone()
        hm.hm_hodlr_factored_adjoint(t, k, U, V, Di, v[0], v[1], 2.0, v[src], gU2, gV2, Di)
        torch.cuda.synchronize()
        check(v[src], gU2, gV2, Di)
    xi, Di = xd.clone(), D.clone()
    hm.hm_hodlr_factored_loss_grad(t, k, U, V, Di, xi, bd, 2.0, xi, r, gx, gU, gV, Di)
    torch.cuda.synchronize()
    assert torch.equal(xi, y)
    check(gx, gU, gV, Di)


@pytest.mark.parametrize("prec", ["fp64", "a32"])
@pytest.mark.parametrize("c", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 119, 120])
def test_panel_widths_recover_exact_rank(prec, c):
    """Panels of c columns (the TSQR and SVD kernels are instantiated per 32 columns)
    on operators of exact rank c - 8 (oversampled by 8: a square Gaussian sample can
    have any condition number), entries small whole numbers so that FP32 holds the
    operator exactly: what is left is rounding, FP64-accurate in both precisions."""
    n, m, p = 1024 + 6, 129, 8 if c > 8 else 0
    f = W.synthetic_hodlr_factors(n, m, c - p, seed=c, shift=0.0)
    rng = np.random.default_rng(c)
    for key in "UV":
        f[key] = [None] + [rng.integers(-2, 3, (n, c - p)).astype(np.float64) for _ in f[key][1:]]
    f["D"] = [np.round(4 * d) for d in f["D"]]
    A = W.dense_from_factors(f)
    At = torch.from_numpy(A).to(DEV, torch.float64 if prec == "fp64" else torch.float32)
    op = hm.hm_dense_operator_create(At, fp64_blocks=prec == "a32", tensor_cores=False)
    h = hm.hm_compress_hodlr(op, hm.Tree(n, m), k=c - p, p=p, seed=7,
                             prec=hm.HM_FP64 if prec == "fp64" else hm.HM_A32)
    err = np.linalg.norm(dense_of(h, n, torch.float64) - A) / np.linalg.norm(A)
    # 1e-16 (2^-46 in double-float sums) times a condition number of about 1e3, three
    # levels deep
    assert err < 1e-9, err
