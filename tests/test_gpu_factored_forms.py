"""The factored layer's forms that only large trees take, with uneven leaves: whole leaves,
gradients in both orders of the tiles, and the fused step's forward with D outside shared
memory and with tiles of 16 rows."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"
U32 = 2.0 ** -24


def layer(n, m, k):
    g = torch.Generator(DEV).manual_seed(n + k)
    t = hm.Tree(n, m)
    nmax = -(-n // 2 ** t.levels)
    U, V = (torch.randn((t.levels, k, n), device=DEV, generator=g) for _ in range(2))
    D = torch.randn((2 ** t.levels, nmax, nmax), device=DEV, generator=g)
    x, b = (torch.randn(n, device=DEV, generator=g) for _ in range(2))
    return t, U, V, D, x, b


class Reference:
    """H x and its adjoint in FP64."""

    def __init__(self, n, m, U, V, D):
        L, start, size = W.tree_ranges(n, m)
        self.L, self.n, self.U, self.V, self.nmax = L, n, U, V, D.shape[1]
        s, z = (torch.as_tensor(np.asarray(v[2 ** L:]), device=DEV) for v in (start, size))
        self.leaf = torch.repeat_interleave(torch.arange(2 ** L, device=DEV), z)
        self.at = self.leaf * self.nmax + torch.arange(n, device=DEV) - s[self.leaf]
        self.live = (torch.arange(self.nmax, device=DEV)[None] < z[:, None])
        self.D = D.double() * self.live[:, None, :] * self.live[:, :, None]

    def leaves(self, x):
        p = torch.zeros(self.live.numel(), device=DEV, dtype=torch.float64)
        p[self.at] = x.double()
        return p.view(-1, self.nmax, 1)

    def project(self, F, x, j):
        node = self.leaf >> (self.L - j)
        p = torch.zeros((2 ** j, F.shape[1]), device=DEV, dtype=torch.float64)
        return p.index_add_(0, node, F[j - 1].T.double() * x.double()[:, None])[node ^ 1]

    def apply(self, x, trans):
        A, B = (self.V, self.U) if trans else (self.U, self.V)
        M = self.D if trans else self.D.transpose(1, 2)  # D is column-major per leaf
        y = torch.bmm(M, self.leaves(x)).view(-1)[self.at]
        for j in range(1, self.L + 1):
            y += (A[j - 1].T.double() * self.project(B, x, j)).sum(1)
        return y

    def adjoint(self, x, r):
        gU, gV = (torch.empty(self.U.shape, device=DEV, dtype=torch.float64) for _ in range(2))
        for j in range(1, self.L + 1):
            gU[j - 1] = (self.project(self.V, x, j) * r.double()[:, None]).T
            gV[j - 1] = (self.project(self.U, r, j) * x.double()[:, None]).T
        return self.apply(r, True), gU, gV, torch.bmm(self.leaves(x), self.leaves(r).transpose(1, 2))


@pytest.mark.parametrize("n,m,k", [(200001, 256, 32),   # apply by whole leaves of 195 and 196
                                   (70001, 256, 8),     # apply and adjoint, of 136 and 137
                                   (50001, 256, 4),     # apply, not transposed, 256 leaves
                                   (130001, 256, 64),   # 576 columns of U beside 254 of D do not fit
                                   (20000, 2, 64)])     # 896 columns of U: tiles of 16 rows
def test_forms_against_fp64(n, m, k):
    t, U, V, D, x, b = layer(n, m, k)
    ref = Reference(n, m, U, V, D)
    mag = Reference(n, m, U.abs(), V.abs(), D.abs())
    # additions on the longest way of a term: within a chunk, over a node's chunks or tiles
    # (several partial sums side by side), over the columns of U and of D
    gamma = (64 + n // 64 + t.levels * k + D.shape[1]) * U32

    def close(got, want, bound, terms=1):
        torch.cuda.synchronize()
        return bool(((got.double() - want).abs() <= terms * gamma * bound).all())

    new = lambda: [torch.full_like(v, float("nan")) for v in (x, U, V, D)]
    for trans in (0, 1):
        y = torch.full_like(x, float("nan"))
        hm.hm_hodlr_factored_apply(t, k, U, V, D, x, y, trans)
        want, bound = ref.apply(x, trans), mag.apply(x.abs(), trans)
        assert close(y, want, bound), trans
        xi = x.clone()
        hm.hm_hodlr_factored_apply(t, k, U, V, D, xi, xi, trans)
        assert close(xi, want, bound), trans
    y, r, g = torch.full_like(x, float("nan")), torch.full_like(x, float("nan")), new()
    hm.hm_hodlr_factored_loss_grad(t, k, U, V, D, x, b, 2.0, y, r, *g)
    want, bound = ref.apply(x, 0), mag.apply(x.abs(), 0) + b.double().abs()
    assert close(y, want, bound) and close(r, want - b.double(), bound)
    wants, bounds = ref.adjoint(x, r), mag.adjoint(x.abs(), r.abs())  # at the step's own r
    for got, w, bd in zip(g, wants, bounds):
        assert close(got, 2 * w, 2 * bd)
    full = new()
    hm.hm_hodlr_factored_adjoint(t, k, U, V, D, x, r, 2.0, *full)
    for got, w, bd in zip(full, wants, bounds):
        assert close(got, 2 * w, 2 * bd)
    for drop in range(1, 15):  # some outputs left out: the others to the bit
        some = [None if drop >> i & 1 else v for i, v in enumerate(new())]
        hm.hm_hodlr_factored_adjoint(t, k, U, V, D, x, r, 2.0, *some)
        torch.cuda.synchronize()
        assert all(a is None or torch.equal(a, f) for a, f in zip(some, full)), drop
        some = [None if drop >> i & 1 else v for i, v in enumerate(new())]
        hm.hm_hodlr_factored_loss_grad(t, k, U, V, D, x, b, 2.0, None, None, *some)
        torch.cuda.synchronize()
        assert all(a is None or torch.equal(a, f) for a, f in zip(some, g)), drop


def test_sixteen_rows_with_d_outside_shared_memory():
    """832 columns of U and leaves of 732: the smallest such tree holds 37 GB of factors.  The
    fused step against the separate calls: each has an error of about u times the square root
    of its longest way of additions (14000 of them), 7e-6 together with the other's 1e-5."""
    n, m, k = 8192 * 731 + 1, 732, 64
    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 40 GB on the device")
    g = torch.Generator(DEV).manual_seed(1)
    t = hm.Tree(n, m)
    U = torch.randn((t.levels, k, n), device=DEV, generator=g)
    D = torch.randn((2 ** t.levels, 732, 732), device=DEV, generator=g)
    x, b = (torch.randn(n, device=DEV, generator=g) for _ in range(2))
    y, r, gx, y2, gx2 = (torch.full_like(x, float("nan")) for _ in range(5))
    hm.hm_hodlr_factored_loss_grad(t, k, U, U, D, x, b, 2.0, y, r, gx)
    hm.hm_hodlr_factored_apply(t, k, U, U, D, x, y2)
    hm.hm_hodlr_factored_adjoint(t, k, U, U, D, x, r, 2.0, gx2)
    torch.cuda.synchronize()
    assert torch.equal(r, y - b)
    for a, c in ((y, y2), (gx, gx2)):
        d, rms = (a - c).double(), float(c.double().square().mean().sqrt())
        assert float(d.square().mean().sqrt()) <= 2e-5 * rms
        assert float(d.abs().max()) <= 1e-3 * rms


@pytest.mark.parametrize("n,m,k", [(70001, 256, 8), (20000, 100, 16)])  # whole leaves, tiles
def test_infinite_factors_stay_infinite(n, m, k):
    """An infinite entry of V, and sums past FP32's range, make their rows of gx infinite (of
    the sign that FP64 gives them), not NaN, and leave the others as they are."""
    t, U, V, D, x, r = layer(n, m, k)
    gx = torch.full_like(x, float("nan"))
    hm.hm_hodlr_factored_adjoint(t, k, U, V, D, x, r, 1.0, gx)
    L = t.levels
    ref = Reference(n, m, U, V, D)
    s = torch.stack([ref.project(U, r, j)[:, c] for j in range(1, L + 1) for c in range(k)])  # U^T r
    Vi, rows = V.clone(), torch.tensor([5, 100, n // 2, n - 1], device=DEV)
    Vi[0, 1, rows[:2]] = float("inf")
    Vi[L - 1, k - 1, rows[2]] = float("-inf")
    Vi[0, 0, rows[3]] = 3e38
    Vi[0, 1, rows[3]] = 3e38 * torch.sign(s[0, rows[3]] * s[1, rows[3]]).float()
    gi = torch.full_like(x, float("nan"))
    hm.hm_hodlr_factored_adjoint(t, k, U, Vi, D, x, r, 1.0, gi)
    torch.cuda.synchronize()
    sign = torch.stack([s[1, 5].sign(), s[1, 100].sign(), -s[-1, n // 2].sign(), s[0, n - 1].sign()])
    assert bool((s[:2, n - 1].abs().sum() * 3e38 > 3.5e38))  # the last row's sum is past the range
    assert torch.equal(gi[rows].double(), sign * float("inf"))
    keep = torch.ones(n, dtype=torch.bool, device=DEV)
    keep[rows] = False
    assert torch.equal(gi[keep], gx[keep])
