"""Gauss-Seidel sweep in the four-colour order where one CTA solves a column (a block's solve and the
scatter of the block before in one launch) against the oracle: one, two and three columns (no
scatter, none, one target), many; one interior node, odd and even meshes, the largest mesh of this
form (n = 89) and the first of the clusters; factors beside the column in shared memory and not
(FP64 from n = 48).  Tolerances: the repository's 1e-12 (FP64) and 1e-6 (FP32) for an application."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,p", [(2, 2, 2), (3, 1, 0), (5, 1, 1), (16, 2, 1), (17, 3, 2), (48, 1, 2),
                                   (64, 2, 2), (89, 1, 2), (90, 1, 2)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_gauss_seidel_sweep(n, M, p, precision):
    prob = O.build_problem(n, M, p, sigma=0.8, ell=0.6)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.8, ell=0.6, precond="fs_gs",
                                         ilu_order="color4", precision=precision))
    R = W.random_field(prob.N, prob.P, seed=41)
    Rd = torch.from_numpy(R).cuda().to(torch.float64 if precision == "fp64" else torch.float32)
    Z = torch.full_like(Rd, float("nan"))
    apply = sg.sg_precond_apply if precision == "fp64" else sg.sg_precond_apply_lowp
    ref = O.fs_precond(prob, Rd.double().cpu().numpy(), mode="gs",
                       blocks=O.fs_blocks(prob, ordering="color4"))
    for _ in range(2):
        apply(h, 0, Rd, Z)
        err = np.abs(Z.double().cpu().numpy() - ref).max() / np.abs(ref).max()
        assert err <= (1e-12 if precision == "fp64" else 1e-6), err
    h.close()
