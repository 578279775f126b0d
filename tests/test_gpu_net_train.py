"""The warm-start network's one-pass training kernel (fixed output layer) at its tile edges."""

import numpy as np
import pytest

from paper_1910_11505_gb300 import sg
from test_gpu_learned import _bf16_round, _unflatten

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B,out,row0", [(128, 132, 0), (256, 1024, 1), (33, 131, 3), (160, 645, 2),
                                        (1, 4096, 1)])
def test_training_pass_tiles_and_alignment(B, out, row0):
    # the one-pass training kernel: unit tiles that end on, before and after a row's copies, batch
    # blocks of 32 rows partly filled, and targets that start 0..3 floats past a 16-byte boundary;
    # reference and tolerance as in test_tensor_core_backprop_matches_reference, the loss as in
    # test_tensor_core_output_layer_matches_reference
    dims = (6, 16, 40, out)
    net = sg.SGNet(*dims, max_batch=256, bf16=True, seed=29)
    rng = np.random.default_rng(9)
    net.set(0, rng.normal(scale=0.4, size=net.num_params).astype(np.float32))
    Z = rng.normal(size=(B, 6)).astype(np.float32)
    T = rng.normal(size=(B, out)).astype(np.float32)
    net.set_basis(torch.from_numpy(T).cuda())
    store = torch.full((B * out + 8,), float("nan"), device="cuda")
    Td = store[row0:row0 + B * out].view(B, out)
    Td.copy_(torch.from_numpy(T))
    Zd = torch.from_numpy(Z).cuda()
    Y = torch.empty(B, out, device="cuda")
    net.forward(Zd, Y)
    loss = net.loss_grad(Zd, Td)
    Yh = Y.cpu().numpy()
    want = float(((Yh.astype(np.float64) - T) ** 2).mean())
    assert abs(loss - want) <= 1e-5 * want
    params = _unflatten(net.get(0), dims)
    W1, b1, W2, b2, W3 = params[:5]
    scale = np.float32(2.0) / (np.float32(B) * np.float32(out))
    dH2 = _bf16_round(scale * (Yh - T)) @ _bf16_round(W3)
    zh = Z.astype(np.float64)
    H1 = np.tanh(zh @ W1.T + b1)
    H2 = np.tanh(H1 @ W2.T + b2)
    dA2 = dH2 * (1.0 - H2 * H2)
    dA1 = (dA2 @ W2) * (1.0 - H1 * H1)
    ref = np.concatenate([(dA1.T @ zh).ravel(), dA1.sum(0), (dA2.T @ H1).ravel(), dA2.sum(0)])
    got = net.get(1).astype(np.float64)[:ref.size]
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    net.close()
