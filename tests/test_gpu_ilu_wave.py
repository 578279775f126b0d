"""Natural-order ILU(0) solves of all columns by warps (mixed systems, mean-based and Jacobi) against
the oracle at the line counts where they can go wrong: the smallest that they serve (12 lines) and one less,
fewer lines than a warp, a warp exactly and one line more, several, the largest (256) and one more.  Tolerance: the
repository's 1e-6 for an FP32 application."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 12, 13, 16, 33, 34, 65, 98, 257, 258])
@pytest.mark.parametrize("pc", ["mean", "fs_jacobi"])
def test_natural_block_solves(n, pc):
    M, p = (2, 2) if n < 60 else (1, 2) if n < 200 else (1, 0)
    prob = O.build_problem(n, M, p, sigma=0.8, ell=0.6)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.8, ell=0.6, precond=pc,
                                         precision="fp32"))
    R = W.random_field(prob.N, prob.P, seed=31)
    Rd = torch.from_numpy(R).cuda().float()
    Z = torch.full_like(Rd, float("nan"))
    sg.sg_precond_apply_lowp(h, 0, Rd, Z)
    Rh = Rd.double().cpu().numpy()
    ref = O.mean_precond(prob, Rh) if pc == "mean" else O.fs_precond(prob, Rh, mode="jacobi")
    err = np.abs(Z.double().cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= 1e-6, err
    h.close()
