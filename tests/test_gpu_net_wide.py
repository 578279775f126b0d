"""The warm-start network's one-pass training kernel with output layers of millions of units."""

import numpy as np
import pytest

from paper_1910_11505_gb300 import sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_rows_of_a_block_more_than_4_gb_apart():
    # 128 rows of 8.5 M targets: row 127 starts 4.3e9 bytes after row 0.  The step over all rows
    # against the mean of the steps over rows 0-63 and 64-127, whose rows lie within 2.2 GB.  A row's
    # dH2 is the same in both (the scale 2 / (B out) differs by a power of two), so the gradients
    # differ by the order of FP32 sums over the batch, 128 x 2^-24 of the terms' sum; the losses by
    # that of 437 tiles x 32 squares per thread, 14 k x 2^-24.
    B, out, dims = 128, 8_500_003, (2, 4, 4)
    net = sg.SGNet(*dims, out, max_batch=B, bf16=True, seed=3)
    gen = torch.Generator(device="cuda").manual_seed(5)
    basis = torch.randn(4, out, generator=gen, device="cuda")
    coef = torch.randn(B, 4, generator=gen, device="cuda") * torch.linspace(0.5, 2, B, device="cuda")[:, None]
    T = coef @ basis
    Z = torch.randn(B, 2, generator=gen, device="cuda")
    net.set_basis(basis)
    ns = net.num_params - 5 * out
    loss, grad = net.loss_grad(Z, T), net.get(1)[:ns].astype(np.float64)
    want, ref = 0.0, np.zeros(ns)
    for rows in (slice(0, 64), slice(64, 128)):
        want += 0.5 * net.loss_grad(Z[rows], T[rows])
        ref += 0.5 * net.get(1)[:ns]
    assert abs(loss - want) <= 1e-3 * want
    assert np.abs(grad - ref).max() <= 1e-4 * np.abs(ref).max()
    net.close()


def test_loss_of_equal_squares():
    # every residual is the same value, so that the rounding of a long FP32 sum does not cancel: 124
    # tiles of 32 squares a thread (4.8e-5 off as one chain of 3968).  FP32 additions on the way of a
    # square: 32 in its tile, 2 for the compensated sum of the tiles, 5 in the warp, 4 over the warps;
    # then two roundings: 45 x 2^-24.
    B, out, dims = 1024, 300_000, (2, 4, 4)
    net = sg.SGNet(*dims, out, max_batch=B, bf16=True, seed=3)
    net.set_basis(torch.zeros(1, out, device="cuda"))  # W3 = 0 (and b3 = 0)
    T = torch.full((B, out), 0.9, device="cuda")
    loss = net.loss_grad(torch.zeros(B, 2, device="cuda"), T)
    want = float(np.float32(0.9)) ** 2
    assert abs(loss - want) <= 45 * 2.0 ** -24 * want
    net.close()
