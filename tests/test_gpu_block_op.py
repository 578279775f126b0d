"""The block-stencil SG operator (the form the automatic choice takes) against the oracle at the
sizes where its tiling can go wrong: one, an odd and an even number of field ranges, padded ranges,
every range size, rows that do not fill the last 32-node tile, meshes of a few nodes, coefficient
degree below 2p, vectors off 16-byte alignment; its use on two streams at once and under capture.

Tolerances: those of the repository's operator tests (1e-12 in FP64, 2e-5 in FP32)."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu

# (n, M, p, q): P and the ranges of fields
CASES = [(3, 3, 2, 0),     # P = 10: 2 ranges of 5; 6 padded rows of one tile
         (5, 2, 4, 0),     # P = 15: 3 ranges of 5
         (9, 5, 2, 3),     # P = 21: 3 ranges of 7, q below 2p
         (12, 6, 2, 0),    # P = 28: 4 ranges of 7
         (33, 3, 3, 0),    # P = 20: 4 ranges of 5
         (16, 4, 3, 0),    # P = 35: 5 ranges of 7
         (6, 5, 3, 0),     # P = 56: 8 ranges of 7
         (4, 6, 3, 0),     # P = 84: 12 ranges of 7
         (160, 2, 1, 0),   # P = 3: one padded range of 4
         (64, 2, 2, 0),    # P = 6: one range of 6
         (100, 1, 6, 0)]   # P = 7: one range of 7


def _setup(case, **kw):
    n, M, p, q = case
    return sg.sg_setup(sg.sg_default_params(n=n, M=M, p=p, q=q, sigma=0.8, ell=0.6, **kw))


def _oracle(case):
    n, M, p, q = case
    return O.build_problem(n, M, p, q=q, sigma=0.8, ell=0.6)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_block_operator_matches_oracle(case, precision):
    h = _setup(case, precision=precision)
    assert sg.sg_op_info(h)[precision]["kernel"] == "block"
    prob = _oracle(case)
    X = W.random_field(prob.N, prob.P, seed=21)
    dt = torch.float64 if precision == "fp64" else torch.float32
    apply = sg.sg_matvec if precision == "fp64" else sg.sg_matvec_lowp
    Xd = torch.from_numpy(X).cuda().to(dt)
    ref = O.sg_matvec(prob, Xd.double().cpu().numpy())
    tol = 1e-12 if precision == "fp64" else 2e-5
    for off in (0, 1):  # the same vectors one element off their alignment
        buf = torch.full((prob.N * prob.P + 2,), float("nan"), dtype=dt, device="cuda")
        src = torch.empty_like(buf)
        src[off:off + Xd.numel()] = Xd.reshape(-1)
        Y = buf[off:off + Xd.numel()].view(prob.N, prob.P)
        apply(h, 0, src[off:off + Xd.numel()].view(prob.N, prob.P), Y)
        err = np.abs(Y.double().cpu().numpy() - ref).max() / np.abs(ref).max()
        assert err <= tol, (off, err)
        assert torch.isnan(buf[:off]).all() and torch.isnan(buf[off + Xd.numel():]).all()
    h.close()


def test_block_operator_in_a_solve_and_levels():
    # alpha, beta and the skipped first product inside GMRES; the operator of every level
    case = (16, 2, 3, 0)
    h = _setup(case, precond="mg", mg_smoother="fg", ilu_order="color4", rtol=1e-12, graphs=1)
    assert sg.sg_op_info(h)["fp64"]["kernel"] == "block"
    prob = _oracle(case)
    F = torch.from_numpy(np.ascontiguousarray(prob.F)).cuda()
    for x0 in (torch.zeros_like(F), torch.ones_like(F)):
        rc, _ = sg.sg_gmres_solve(h, [F], [x0])
        r = prob.F - O.sg_matvec(prob, x0.cpu().numpy())
        assert rc == sg.SG_OK and np.linalg.norm(r) <= 2e-12 * np.linalg.norm(prob.F)
    h.close()


def test_block_operator_on_two_streams_and_captured():
    case = (64, 4, 3, 0)
    h = _setup(case)
    N, P, _ = sg.sg_dims(h)
    X = [torch.from_numpy(W.random_field(N, P, seed=s)).cuda() for s in (1, 2)]
    want = [torch.empty_like(x) for x in X]
    for x, y in zip(X, want):
        sg.sg_matvec(h, 0, x, y)
    torch.cuda.synchronize()
    Y = [torch.full_like(x, float("nan")) for x in X]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(20):
        for s, x, y in zip(streams, X, Y):
            sg.sg_matvec(h, 0, x, y, stream=s)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(Y, want))
    g = torch.cuda.CUDAGraph()
    Y[0].fill_(float("nan"))
    with torch.cuda.graph(g):
        sg.sg_matvec(h, 0, X[0], Y[0])
    for _ in range(2):
        Y[0].fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(Y[0], want[0])
    del g
    h.close()
