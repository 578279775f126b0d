"""Colour phases of the grouped field split at the thread layouts where they can go wrong: splits of
1, 4, 6, 10, 21 and 35 fields (several nodes per CTA, unit columns that do not divide by the groups,
fields that are no multiple of four in BF16), meshes from one interior node to more nodes than the
grouping threshold, against the oracle.  Tolerances are the repository's for a grouped-split
application: 1e-12 in FP64, 1e-5 max(1, Q / 8) in FP32; BF16 factors add 2^-8 of the result."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M,p", [(2, 2, 2), (3, 5, 2), (7, 4, 3), (24, 2, 0), (40, 3, 1), (24, 2, 2),
                                   (10, 3, 2)])
@pytest.mark.parametrize("form", ["fp64", "fp32", "bf16"])
def test_phases_match_oracle(n, M, p, form):
    prob = O.build_problem(n, M, p, sigma=0.7, ell=0.6)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.7, ell=0.6, precond="fg",
                                         fg_rule="whole", ilu_order="color4",
                                         precision="fp64" if form == "fp64" else "fp32",
                                         fg_bf16=int(form == "bf16")))
    dt = torch.float64 if form == "fp64" else torch.float32
    R = torch.from_numpy(W.random_field(prob.N, prob.P, seed=41)).cuda().to(dt)
    Z = torch.full_like(R, float("nan"))
    (sg.sg_precond_apply if form == "fp64" else sg.sg_precond_apply_lowp)(h, 0, R, Z)
    splits = [(0, prob.P)]
    ref = O.fg_precond(prob, R.double().cpu().numpy(), splits, O.fg_blocks(prob, splits, "color4"))
    err = np.abs(Z.double().cpu().numpy() - ref).max() / np.abs(ref).max()
    tol = 1e-12 if form == "fp64" else 1e-5 * max(1, prob.P / 8)
    if form == "bf16":
        tol += 4 * 2.0 ** -8  # eight roundings of a half unit along the forward and backward phases
    assert err <= tol, err
    h.close()
