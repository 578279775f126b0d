"""The block-stencil operator with 18 to 30 ranges of fields, where one CTA fills its SM and the ring
has to leave room for the staged differences.  Reference: the pair kernel (tested against the oracle,
which takes minutes at these basis sizes); tolerances of the operator tests, 1e-12 and 2e-5."""

import pytest

from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,M,p,P", [(9, 4, 5, 126), (33, 4, 5, 126), (7, 8, 3, 165), (8, 4, 6, 210)])
def test_block_operator_of_wide_bases(n, M, p, P, precision):
    kw = dict(n=n, M=M, p=p, sigma=0.8, ell=0.6, precond="none", restart=2)
    h = sg.sg_setup(sg.sg_default_params(precision=precision, **kw))
    assert sg.sg_op_info(h)[precision]["kernel"] == "block"
    ref = sg.sg_setup(sg.sg_default_params(op_kernel="pairs", **kw))
    N = (n + 1) ** 2
    dt = torch.float64 if precision == "fp64" else torch.float32
    apply = sg.sg_matvec if precision == "fp64" else sg.sg_matvec_lowp
    X = torch.from_numpy(W.random_field(N, P, seed=7)).cuda().to(dt)
    Y = torch.full_like(X, float("nan"))
    apply(h, 0, X, Y)
    want = torch.empty(N, P, dtype=torch.float64, device="cuda")
    sg.sg_matvec(ref, 0, X.double(), want)
    err = (Y.double() - want).abs().max() / want.abs().max()
    assert float(err) <= (1e-12 if precision == "fp64" else 2e-5)
    h.close()
    ref.close()
