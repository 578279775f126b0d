"""The automatic operator choice at coefficient degrees below 2p, where the sparse forms' work falls
under the block-stencil form's."""

import numpy as np
import pytest

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _setup(n, M, p, q, precision, **kw):
    return sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, q=q, sigma=0.8, ell=0.6, precond="none", restart=2,
                                            precision=precision, **kw))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,M,p,q,kinds", [
    (20, 6, 3, 1, ("pairs", "tile")),           # 0.11 of the block form's multiply-adds
    (40, 4, 3, 1, ("pairs", "tile")),           # 0.22
    (20, 4, 3, 2, ("pairs", "tile", "block")),  # 0.64: timed
    (20, 4, 3, 4, ("block",)),                  # 2.03
    (20, 4, 3, 0, ("block",))])                 # 3.35
def test_operator_choice_by_coefficient_degree(n, M, p, q, kinds, precision):
    h, again = (_setup(n, M, p, q, precision) for _ in range(2))
    info = [sg.sg_op_info(x) for x in (h, again)]
    assert info[0][precision]["kernel"] in kinds, info[0]
    assert info[1][precision]["kernel"] == info[0][precision]["kernel"]
    if kinds != ("block",):
        assert "cached" in info[1]["msg"], info[1]
    prob = O.build_problem(n, M, p, q=q, sigma=0.8, ell=0.6)
    dt = torch.float64 if precision == "fp64" else torch.float32
    apply = sg.sg_matvec if precision == "fp64" else sg.sg_matvec_lowp
    X = torch.from_numpy(W.random_field(prob.N, prob.P, seed=5)).cuda().to(dt)
    Y = torch.full_like(X, float("nan"))
    apply(h, 0, X, Y)
    ref = O.sg_matvec(prob, X.double().cpu().numpy())
    err = np.abs(Y.double().cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= (1e-12 if precision == "fp64" else 2e-5)
    h.close()
    again.close()
