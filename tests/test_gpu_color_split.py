"""Four-colour block solves with the column in the shared memory of a cluster against the oracle: the
smallest meshes of each cluster size (2, 4, 8 and 16 CTAs), odd and even ones, a last CTA with few
lines; single columns (Gauss-Seidel, coupled) and several; and a mesh beyond that form (its lines
take more than 200 KB).  Tolerances: the repository's 1e-12 (FP64) and 1e-6 (FP32) for an
application."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,pc", [(90, "fs_gs"), (91, "mean"), (126, "fs_gs"), (127, "fs_gs"), (128, "fs_gs"),
                                  (129, "fs_jacobi"), (180, "fs_gs"), (181, "fs_gs"), (200, "mean"),
                                  (256, "fs_gs"), (270, "fs_gs"), (460, "mean")])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_color_solves(n, pc, precision):
    M, p = (1, 2) if n < 200 else (1, 1)
    prob = O.build_problem(n, M, p, sigma=0.8, ell=0.6)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.8, ell=0.6, precond=pc,
                                         ilu_order="color4", precision=precision))
    R = W.random_field(prob.N, prob.P, seed=43)
    Rd = torch.from_numpy(R).cuda().to(torch.float64 if precision == "fp64" else torch.float32)
    Z = torch.full_like(Rd, float("nan"))
    (sg.sg_precond_apply if precision == "fp64" else sg.sg_precond_apply_lowp)(h, 0, Rd, Z)
    Rh = Rd.double().cpu().numpy()
    if pc == "mean":
        ref = O.mean_precond(prob, Rh, ordering="color4")
    else:
        ref = O.fs_precond(prob, Rh, mode=pc[3:], blocks=O.fs_blocks(prob, ordering="color4"))
    err = np.abs(Z.double().cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= (1e-12 if precision == "fp64" else 1e-6), err
    h.close()
