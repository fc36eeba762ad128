"""A call's result does not depend on how the lanes of its kernels are scheduled: the
same compression again gives the same bits (the panel QR and SVD kernels let 8-lane
groups read and update shared norms and rows between block barriers)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
hm = pytest.importorskip("paper_1503_07152_gb300")
DEV = "cuda:0"


@pytest.mark.parametrize("prec", ["fp64", "mixed", "a32"])
@pytest.mark.parametrize("n,m,r", [(515, 33, 13), (1030, 65, 24), (2048, 128, 60)])
def test_repeated_compressions_give_the_same_bits(prec, n, m, r):
    A = torch.from_numpy(W.log_kernel(n).astype(np.float64))
    At = A.to(DEV, torch.float64 if prec == "fp64" else torch.float32)
    op = hm.hm_dense_operator_create(At, fp64_blocks=prec == "a32")
    p = {"fp64": hm.HM_FP64, "mixed": hm.HM_MIXED, "a32": hm.HM_A32}[prec]
    t = hm.Tree(n, m)
    dt = torch.float32 if prec == "mixed" else torch.float64

    def factors():
        h = hm.hm_compress_hodlr(op, t, k=r - 4, p=4, seed=2, prec=p)
        out = torch.empty((2, t.levels, h.info["r"], n), device=DEV, dtype=dt)
        for lv in range(1, t.levels + 1):
            hm.hm_hodlr_export_level(h, lv, out[0, lv - 1], out[1, lv - 1])
        torch.cuda.synchronize()
        return out

    first = factors()
    for _ in range(6):
        assert torch.equal(first, factors())
