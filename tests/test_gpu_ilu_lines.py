"""Natural-order ILU(0) solves by warps in FP64 (mean-based, Jacobi and Gauss-Seidel) against the oracle
at the line counts where they can go wrong: the smallest that they serve (12 lines) and one less,
fewer lines than a warp's 16, a warp exactly and one line more, an even line count (the column's odd stride), the largest column that shared
memory holds and one more.  Tolerance: the repository's 1e-12 for an FP64 application."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 12, 13, 17, 18, 33, 35, 66, 97, 128, 130, 131, 132, 133, 134])
@pytest.mark.parametrize("pc", ["mean", "fs_jacobi", "fs_gs"])
def test_natural_block_solves(n, pc):
    M, p = (2, 2) if n < 60 else (1, 2)
    prob = O.build_problem(n, M, p, sigma=0.8, ell=0.6)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.8, ell=0.6, precond=pc))
    R = W.random_field(prob.N, prob.P, seed=37)
    Rd = torch.from_numpy(R).cuda()
    Z = torch.full_like(Rd, float("nan"))
    sg.sg_precond_apply(h, 0, Rd, Z)
    ref = O.mean_precond(prob, R) if pc == "mean" else O.fs_precond(prob, R, mode=pc[3:])
    err = np.abs(Z.cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= 1e-12, err
    h.close()
