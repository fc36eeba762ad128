"""The panel kernels (TSQR, SVD, CholQR) at each width, to their own precision: FP64, and
double-float sums for HM_A32."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import hodlr as ohodlr
from oracle.tree import build_tree

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"


@pytest.mark.parametrize("c", [1, 2, 17, 31, 32, 33, 48, 63, 64, 65, 96, 97, 119, 120])
def test_panels_to_their_precision(c):
    """An operator of exact rank that FP32 holds exactly, so that rounding is all that is left.
    The FP64 oracle with the same test matrices shows what rounding costs on this operator;
    16 times that is allowed for FP64, and 2^8 times more for double-float operations (2^-45
    against 2^-53).  The bases are orthonormal to 16 c units of either."""
    n, m, p = 1030, 129, 8 if c > 8 else 0
    k = c - p
    f = W.synthetic_hodlr_factors(n, m, k, seed=c, shift=0.0)
    rng = np.random.default_rng(c)
    for key in "UV":
        f[key] = [None] + [rng.integers(-2, 3, (n, k)).astype(np.float64) for _ in f[key][1:]]
    f["D"] = [np.round(4 * d) for d in f["D"]]
    A = W.dense_from_factors(f)
    tree = build_tree(n, m)
    o = ohodlr.compress(ohodlr.dense_apply_fn(A), tree, r=c, k=k, seed=7)
    rounding = np.linalg.norm(ohodlr.dense(o) - A) / np.linalg.norm(A)
    for prec, unit in (("fp64", 1.0), ("a32", 2.0 ** 8)):
        At = torch.from_numpy(A).to(DEV, torch.float64 if prec == "fp64" else torch.float32)
        op = hm.hm_dense_operator_create(At, fp64_blocks=prec == "a32", tensor_cores=False)
        t = hm.Tree(n, m)
        h = hm.hm_compress_hodlr(op, t, k=k, p=p, seed=7, prec=hm.HM_FP64 if prec == "fp64" else hm.HM_A32)
        out = torch.empty((n, n), device=DEV, dtype=torch.float64)
        hm.hm_reconstruct_block(h, 0, n, 0, n, out)
        torch.cuda.synchronize()
        err = np.linalg.norm(out.cpu().numpy().T - A) / np.linalg.norm(A)
        assert err <= 16 * unit * rounding, (prec, err, rounding)
        L, start, size = W.tree_ranges(n, m)
        for lv in range(1, L + 1):
            U, V = (torch.empty((h.info["r"], n), device=DEV, dtype=torch.float64) for _ in range(2))
            hm.hm_hodlr_export_level(h, lv, U, V)
            V = V.cpu().numpy()
            for node in range(2 ** lv, 2 ** (lv + 1)):
                Q = V[:k, start[node]:start[node] + size[node]]
                assert np.linalg.norm(Q @ Q.T - np.eye(k), 2) <= 16 * c * unit * 2.0 ** -53, (prec, lv, node)
