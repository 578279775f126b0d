"""Paths that an application meets only when something has gone wrong, entered on purpose on the host."""

import numpy as np
import pytest

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _hook(what, value):
    assert sg.load_library().sg_test_hook(what, sg.ctypes.c_longlong(value)) == sg.SG_OK


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,M,p", [(40, 4, 3), (12, 6, 3), (60, 3, 2)])
def test_block_operator_waits_that_give_up(n, M, p, precision):
    # every CTA goes on as after a wait that was given up: interior rows are NaN, boundary rows are X, the
    # kernel ends, and the next call is right (several items per CTA, rings shorter and longer than an
    # item's tiles, odd and even numbers of ranges)
    h = sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, sigma=0.8, ell=0.6, precision=precision))
    assert sg.sg_op_info(h)[precision]["kernel"] == "block"
    prob = O.build_problem(n, M, p, sigma=0.8, ell=0.6)
    dt = torch.float64 if precision == "fp64" else torch.float32
    apply = sg.sg_matvec if precision == "fp64" else sg.sg_matvec_lowp
    X = torch.from_numpy(W.random_field(prob.N, prob.P, seed=3)).cuda().to(dt)
    Y = torch.zeros_like(X)
    try:
        _hook(0, 1)
        apply(h, 0, X, Y)
        torch.cuda.synchronize()
    finally:
        _hook(0, 0)
    inner = torch.zeros(n + 1, n + 1, dtype=torch.bool, device="cuda")
    inner[1:-1, 1:-1] = True
    inner = inner.reshape(-1)
    assert torch.isnan(Y[inner]).all() and torch.equal(Y[~inner], X[~inner])
    apply(h, 0, X, Y)
    ref = O.sg_matvec(prob, X.double().cpu().numpy())
    assert np.abs(Y.double().cpu().numpy() - ref).max() <= (1e-12 if precision == "fp64" else 2e-5) * np.abs(ref).max()
    h.close()
