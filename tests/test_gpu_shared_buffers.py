"""Outputs that share memory with inputs: the factored layer's calls and the handles' where
the header allows it, at shifts that make a block's output another block's input, give
what they give with buffers of their own."""
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"


def layer(n, m, k):
    g = torch.Generator(DEV).manual_seed(n + k)
    t = hm.Tree(n, m)
    nmax = -(-n // 2 ** t.levels)
    U, V = (torch.randn((t.levels, k, n), device=DEV, generator=g) for _ in range(2))
    D = torch.randn((2 ** t.levels, nmax, nmax), device=DEV, generator=g)
    x, b = (torch.randn(n, device=DEV, generator=g) for _ in range(2))
    return t, U, V, D, x, b


def pair(x, d):
    """One buffer and two views of it, the first holding x, the second d entries on."""
    n = x.numel()
    buf = torch.full((n + abs(d),), float("nan"), device=DEV)
    a, c = (buf[:n], buf[d:]) if d >= 0 else (buf[-d:], buf[:n])
    a.copy_(x)
    return a, c


# the last two take the whole-leaf kernels (the adjoint's: the last)
SIZES = [(515, 33, 9), (4096, 256, 32), (5003, 64, 5), (200001, 256, 32), (70001, 256, 8)]


@pytest.mark.parametrize("n,m,k", SIZES)
def test_apply_over_part_of_x(n, m, k):
    t, U, V, D, x, _ = layer(n, m, k)
    for trans in (0, 1):
        want = torch.full_like(x, float("nan"))
        hm.hm_hodlr_factored_apply(t, k, U, V, D, x, want, trans)
        for d in (1, -1, 100, -(n // 2), n - 1):
            for call in (hm.hm_hodlr_factored_apply, hm.hm_hodlr_factored_apply_noalloc):
                a, y = pair(x, d)
                call(t, k, U, V, D, a, y, trans)
                torch.cuda.synchronize()
                assert torch.equal(y, want), (trans, d)


def test_noalloc_copy_of_x_beyond_its_scratch_is_refused():
    # 1 MB of projections, and the 8.8 MB copy of x, against the 8 MiB buffer
    t, U, V, D, x, _ = layer(2200000, 64, 1)
    a, y = pair(x, 1)
    hm.hm_hodlr_factored_apply(t, 1, U, V, D, x, torch.empty_like(x))  # uploads the tree
    with pytest.raises(hm.HmError, match="scratch"):
        hm.hm_hodlr_factored_apply_noalloc(t, 1, U, V, D, a, y)
    hm.hm_hodlr_factored_apply_noalloc(t, 1, U, V, D, a, a)  # y = x needs no copy
    torch.cuda.synchronize()
    assert torch.isfinite(a).all()


@pytest.mark.parametrize("n,m,k", SIZES)
def test_gradients_over_inputs(n, m, k):
    t, U, V, D, x, b = layer(n, m, k)
    new = lambda: [torch.full_like(v, float("nan")) for v in (x, U, V, D)]

    def same(got, want):
        torch.cuda.synchronize()
        return all(torch.equal(g, w) for g, w in zip(got, want))

    want = new()
    hm.hm_hodlr_factored_adjoint(t, k, U, V, D, x, b, 2.0, *want)
    for d in (0, 1, -100):  # gx over x, over r
        for src in (0, 1):
            a, gx = pair((x, b)[src], d)
            out = [gx] + new()[1:]
            hm.hm_hodlr_factored_adjoint(t, k, U, V, D, *((a, b) if src == 0 else (x, a)), 2.0, *out)
            assert same(out, want), (d, src)
    Ui, Vi, Di = U.clone(), V.clone(), D.clone()  # every gradient in its factor's place
    out = [new()[0], Ui, Vi, Di]
    hm.hm_hodlr_factored_adjoint(t, k, Ui, Vi, Di, x, b, 2.0, *out)
    assert same(out, want)

    y, r = torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
    want = new()
    hm.hm_hodlr_factored_loss_grad(t, k, U, V, D, x, b, 2.0, y, r, *want)
    step = lambda x_, b_, y_, r_, out, U_=U, V_=V, D_=D: \
        hm.hm_hodlr_factored_loss_grad(t, k, U_, V_, D_, x_, b_, 2.0, y_, r_, *out)
    ny, nr = torch.empty_like(y), torch.empty_like(r)
    for d in (0, 1, -100):
        for src in (0, 1):  # y, r and gx over x, over b
            v = (x, b)[src]
            args = lambda a: (a, b) if src == 0 else (x, a)
            a, o = pair(v, d)
            out = new()
            step(*args(a), o, nr, out)
            assert same([o, nr, *out], [y, r, *want]), ("y", d, src)
            a, o = pair(v, d)
            out = new()
            step(*args(a), ny, o, out)
            assert same([ny, o, *out], [y, r, *want]), ("r", d, src)
            a, o = pair(v, d)
            out = [o] + new()[1:]
            step(*args(a), ny, nr, out)
            assert same([ny, nr, *out], [y, r, *want]), ("gx", d, src)
        a, o = pair(x, d)  # gx over r
        out = [o] + new()[1:]
        step(x, b, ny, a, out)
        assert same([ny, *out], [y, *want]), ("gx over r", d)
    Ui, Vi, Di = U.clone(), V.clone(), D.clone()
    out = [new()[0], Ui, Vi, Di]
    step(x, b, ny, nr, out, Ui, Vi, Di)
    assert same([ny, nr, *out], [y, r, *want])
    Vi = V.clone()  # gU in V's place
    out = [new()[0], Vi, *new()[2:]]
    step(x, b, ny, nr, out, U, Vi, D)
    assert same([ny, nr, *out], [y, r, *want])


def handle(kind, n):
    A = torch.from_numpy(W.log_kernel(n)).to(DEV, torch.float32 if kind == "mixed" else torch.float64)
    A += float(n) * torch.eye(n, device=DEV, dtype=A.dtype)
    op, t = hm.hm_dense_operator_create(A), hm.Tree(n, 65)
    if kind == "hbsid":
        return hm.hm_compress_hbs(op, t, tol=1e-6, r=24, seed=2, prec=hm.HM_FP64)
    return hm.hm_compress_hodlr(op, t, k=16, p=4, seed=2, prec=hm.HM_MIXED if kind == "mixed" else hm.HM_FP64)


@pytest.mark.parametrize("kind", ["fp64", "mixed", "hbsid"])
@pytest.mark.parametrize("c", [1, 3, 128, 129, 300])
def test_blocks_that_share_memory(kind, c):
    """hm_apply and hm_solve with Y (X) at shifts by rows and columns over X (B), at other
    leading dimensions and in X's place, past the 128 columns that go together."""
    n = 515
    h = handle(kind, n)
    dt = torch.float32 if kind == "mixed" else torch.float64
    X = torch.randn((c, n), device=DEV, dtype=dt, generator=torch.Generator(DEV).manual_seed(c))
    calls = [hm.hm_apply]
    if kind != "hbsid":
        hm.hm_hodlr_factorize(h)
        calls.append(hm.hm_solve)
    for call in calls:
        for trans in (0, 1):
            want = torch.full_like(X, float("nan"))
            call(h, trans, X, want)
            for ldx, ldy, off in ((n, n, 0), (n + 7, n, 0), (n, n + 7, 0), (n, n, n), (n, n, -n), (n, n, 1),
                                  (n, n + 1, -5), (2 * n, 2 * n, n), (2 * n, 2 * n, n - 1), (n, 2 * n, n),
                                  (n, n, (c // 2) * n)):
                buf = torch.full(((c + 1) * 2 * n + abs(off) + 8 * c,), float("nan"), device=DEV, dtype=dt)
                x0 = max(0, -off)
                a = torch.as_strided(buf, (c, n), (ldx, 1), x0)
                y = torch.as_strided(buf, (c, n), (ldy, 1), x0 + off)
                a.copy_(X)
                call(h, trans, a, y)
                torch.cuda.synchronize()
                assert torch.equal(y, want), (call.__name__, trans, ldx, ldy, off)
