"""Arnoldi steps on one cluster (short vectors) and on the whole GPU (longer ones), and both back
substitutions, against the oracle's GMRES: vectors of 54 entries (slices shorter than a warp, the
last ones empty), either side of the 32 768-entry limit, cycles of one step and beyond 128 steps.

A solve to 1e-10 stops within one iteration of the oracle's count (the repository's criterion for
GMRES) with a true residual within 1.5 of the tolerance."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,p,restart", [(2, 2, 2, 30), (5, 1, 2, 1), (16, 2, 2, 30),
                                           (72, 2, 2, 300), (74, 2, 2, 300)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_solve_matches_oracle_gmres(n, M, p, restart, precision):
    prob = O.build_problem(n, M, p, sigma=0.5, ell=1.0)
    rtol, cap = 1e-10, (200 if restart == 1 else 400)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.5, ell=1.0, precond="mean",
                                         restart=restart, rtol=rtol, max_iters=cap,
                                         precision=precision))
    F = torch.from_numpy(np.ascontiguousarray(prob.F)).cuda()
    x = torch.zeros_like(F)
    rc, info = sg.sg_gmres_solve(h, [F], [x])
    h.close()
    res = np.linalg.norm(prob.F - O.sg_matvec(prob, x.cpu().numpy())) / np.linalg.norm(prob.F)
    assert rc == sg.SG_OK and res <= 1.5 * rtol, (rc, info, res)
    if precision == "fp64":
        LU = O.ilu0(prob.A[0])
        _, ref = O.gmres(lambda v: O.sg_matvec(prob, v.reshape(prob.N, prob.P)).ravel(),
                         lambda v: O.mean_precond(prob, v.reshape(prob.N, prob.P), LU=LU).ravel(),
                         prob.F.ravel(), restart=restart, rtol=rtol, max_iters=cap)
        assert abs(info[0]["iters"] - ref["iters"]) <= 1, (info[0]["iters"], ref["iters"])
