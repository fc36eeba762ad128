"""The solver's pivots are inverted to the last bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"


def values(n):
    """Fractions at random, next to 1 and next to 2 (and all ones), at exponents over nearly
    the whole range and at its ends, both signs."""
    rng = np.random.default_rng(5)
    frac = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    frac[: n // 4] = np.arange(n // 4, dtype=np.uint64)
    frac[n // 4: n // 2] = ((1 << 52) - 1) - np.arange(n // 4, dtype=np.uint64)
    exp = rng.integers(60, 1987, n)
    exp[::3] = rng.integers(1003, 1044, exp[::3].size)
    frac[7::16] = (1 << 52) - 1
    return (frac | (exp.astype(np.uint64) << np.uint64(52)) |
            (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63))).view(np.float64)


def test_diagonal_leaves_are_inverted_to_the_bit():
    """A diagonal operator: its inverse's entries are the reciprocals of its own, and a
    product with ones adds nothing but zeros to them."""
    n = 2048
    x = values(n)
    A = torch.diag(torch.from_numpy(x)).to(DEV)
    h = hm.hm_compress_hodlr(hm.hm_dense_operator_create(A), hm.Tree(n, 200), k=2, p=2, seed=1, prec=hm.HM_FP64)
    hm.hm_hodlr_factorize(h)
    B = torch.ones((1, n), device=DEV, dtype=torch.float64)
    for trans in (0, 1):
        X = torch.empty_like(B)
        hm.hm_solve(h, trans, B, X)
        torch.cuda.synchronize()
        assert np.array_equal(X.cpu().numpy()[0], 1.0 / x)
