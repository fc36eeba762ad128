"""The FP64 sums of the handles' products: formed over 16 terms at a time (shorter chains
round less), in an order that does not depend on how many columns go along."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"
LD = np.longdouble


def fma(a, b, c):
    """a b + c rounded once (a long double holds the product of two doubles)."""
    return (a.astype(LD) * b + c).astype(np.float64)


def chain(A, B, groups):
    """sum_k A[:, k] B[k], each group of k a chain of FMAs, the groups' sums added in turn."""
    acc = np.zeros((A.shape[0], B.shape[1]))
    for g in groups:
        t = np.zeros_like(acc)
        for k in g:
            t = fma(A[:, k:k + 1], B[k:k + 1], t)
        acc = acc + t
    return acc


def cut(n, step):
    return [range(i, min(n, i + step)) for i in range(0, n, step)]


def compressed(n, m, k, prec):
    A = W.dense_from_factors(W.synthetic_hodlr_factors(n, m, k, seed=n, shift=float(n)))
    At = torch.from_numpy(A).to(DEV, torch.float64 if prec == "fp64" else torch.float32)
    op = hm.hm_dense_operator_create(At, fp64_blocks=prec == "a32")
    p = {"fp64": hm.HM_FP64, "mixed": hm.HM_MIXED, "a32": hm.HM_A32}[prec]
    t = hm.Tree(n, m)
    return t, hm.hm_compress_hodlr(op, t, k=k, p=4, seed=2, prec=p)


@pytest.mark.skipif(np.finfo(LD).nmant < 105, reason="a long double does not hold a product of doubles")
@pytest.mark.parametrize("n,m,k", [(1100, 140, 17), (1536, 200, 40)])
def test_apply_sums_sixteen_terms_at_a_time(n, m, k):
    t, h = compressed(n, m, k, "fp64")
    L, r = t.levels, h.info["r"]
    f = W.tree_ranges(n, m)
    start, size = (np.asarray(v) for v in f[1:])
    U, V = (torch.empty((L, r, n), device=DEV, dtype=torch.float64) for _ in range(2))
    for lv in range(1, L + 1):
        hm.hm_hodlr_export_level(h, lv, U[lv - 1], V[lv - 1])
    U, V = (v.cpu().numpy() for v in (U, V))
    X = np.random.default_rng(n).standard_normal((n, 3))
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).to(DEV)
    Yd = torch.empty_like(Xd)
    hm.hm_apply(h, 0, Xd, Yd)
    torch.cuda.synchronize()
    want = np.empty_like(X)
    for node in range(2 ** L, 2 ** (L + 1)):  # the leaves: four chains of 32 of every 128 columns
        s, z = int(start[node]), int(size[node])
        D = torch.empty((z, z), device=DEV, dtype=torch.float64)
        hm.hm_reconstruct_block(h, s, s + z, s, s + z, D)
        D = D.cpu().numpy().T
        parts = [chain(D, X[s:s + z], [[k for k in range(z) if k // 32 % 4 == w]]) for w in range(4)]
        want[s:s + z] = ((parts[0] + parts[1]) + parts[2]) + parts[3]
    for lv in range(1, L + 1):
        coef = {}
        for node in range(2 ** lv, 2 ** (lv + 1)):  # chunks of at most 256 rows, then their sum
            s, z = int(start[node]), int(size[node])
            coef[node] = np.zeros((r, 3))
            for c in cut(z, 256):
                rows = slice(s + c[0], s + c[-1] + 1)
                coef[node] = coef[node] + chain(V[lv - 1][:, rows], X[rows], cut(len(c), 16))
        for node in range(2 ** lv, 2 ** (lv + 1)):
            s, z = int(start[node]), int(size[node])
            want[s:s + z] += chain(U[lv - 1][:, s:s + z].T, coef[node ^ 1], cut(r, 16))
    assert np.array_equal(Yd.cpu().numpy().T, want)


COLS = [1, 2, 5, 8, 9, 31, 33, 64, 65, 100, 128, 129, 150]


@pytest.mark.parametrize("prec", ["fp64", "mixed", "a32"])
@pytest.mark.parametrize("n,m,k", [(1100, 140, 17), (6000, 100, 60)])
def test_a_column_alone_and_among_others(prec, n, m, k):
    """hm_apply and hm_solve: the same bits for a column whatever goes along with it."""
    t, h = compressed(n, m, k, prec)
    hm.hm_hodlr_factorize(h)
    dt = torch.float32 if prec == "mixed" else torch.float64
    X = torch.randn((max(COLS), n), device=DEV, dtype=dt, generator=torch.Generator(DEV).manual_seed(k))
    for call in (hm.hm_apply, hm.hm_solve):
        for trans in (0, 1):
            full = torch.empty_like(X)
            call(h, trans, X, full)
            for c in COLS:
                Y = torch.empty_like(X[:c])
                call(h, trans, X[:c], Y)
                torch.cuda.synchronize()
                assert torch.equal(Y, full[:c]), (call.__name__, trans, c)


@pytest.mark.parametrize("n", [4000, 20001])
def test_a_column_alone_and_among_others_hbsid(n):
    op = hm.hm_log_kernel_operator_create(n)
    h = hm.hm_compress_hbs(op, hm.Tree(n, 256), tol=1e-7, r=60, seed=3, prec=hm.HM_A32)
    X = torch.randn((max(COLS), n), device=DEV, dtype=torch.float64,
                    generator=torch.Generator(DEV).manual_seed(n))
    for trans in (0, 1):
        full = torch.empty_like(X)
        hm.hm_apply(h, trans, X, full)
        for c in COLS:
            Y = torch.empty_like(X[:c])
            hm.hm_apply(h, trans, X[:c], Y)
            torch.cuda.synchronize()
            assert torch.equal(Y, full[:c]), (trans, c)


def dense(n, kind, seed=0):
    A = np.random.default_rng(n + seed).standard_normal((n, n)).astype(np.float32).astype(np.float64)
    At = torch.from_numpy(A).to(DEV, torch.float64 if kind == "fp64" else torch.float32)
    return A, hm.hm_dense_operator_create(At, fp64_blocks=kind == "a32", tensor_cores=False)


@pytest.mark.parametrize("kind", ["fp64", "a32"])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 100, 150, 1100, 4100, 16100])
def test_dense_column_alone_and_among_others(kind, n):
    """One to eight blocks a tile (by n); columns that share their 32 with zeros elsewhere."""
    _, op = dense(n, kind)
    X = torch.randn((max(COLS), n), device=DEV, dtype=torch.float64, generator=torch.Generator(DEV).manual_seed(n))
    X[::3, : n // 2] = 0.0
    X[1::3, n // 3:] = 0.0
    for trans in (0, 1):
        full = torch.empty_like(X)
        hm.hm_dense_apply(op, trans, X, full)
        for c in COLS + [-1, -7]:  # the first columns, or a few from the end
            part = slice(0, c) if c > 0 else slice(c, None)
            Y = torch.empty_like(X[part])
            hm.hm_dense_apply(op, trans, X[part], Y)
            torch.cuda.synchronize()
            assert torch.equal(Y, full[part]), (trans, c)


@pytest.mark.parametrize("kind", ["fp64", "a32"])
@pytest.mark.parametrize("n", [1000, 8192, 16400])
def test_dense_products_round_as_sums_of_sixteen(kind, n):
    """The rounding error, against that of products summed 16 at a time and those sums added
    up one by one (emulated on the same data): not above it, with 10% for the scatter of
    1024 errors (3%) and the emulation's rounded products (2%)."""
    rows = np.random.default_rng(1).choice(n, 256, replace=False)
    A, op = dense(n, kind)
    X = np.random.default_rng(2).standard_normal((n, 4))
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).to(DEV)
    for trans in (0, 1):
        Y = torch.empty_like(Xd)
        hm.hm_dense_apply(op, trans, Xd, Y)
        torch.cuda.synchronize()
        M = (A.T if trans else A)[rows]
        # exact sums: the entries of A have 24 bits and X is cut in two of 27 and 26, so the
        # products are exact, and the error-free running sum keeps what each addition loses
        Xh = (X.astype(np.float32)).astype(np.float64)
        hi, lo, emul, t = (np.zeros((256, 4)) for _ in range(4))
        for k in range(n):
            for part in (Xh[k], X[k] - Xh[k]):
                p = M[:, k:k + 1] * part
                s = hi + p
                z = s - hi
                lo += (hi - (s - z)) + (p - z)
                hi = s
            t = t + M[:, k:k + 1] * X[k]
            if k % 16 == 15 or k == n - 1:
                emul, t = emul + t, np.zeros_like(t)
        rms = lambda y: np.sqrt(np.mean(((y - hi) - lo) ** 2))
        assert rms(Y.cpu().numpy().T[rows]) <= 1.1 * rms(emul), trans
