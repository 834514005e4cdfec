"""The network's kernels on ragged images and on more tiles than blocks.

The convolutions work on 16 x 16 tiles with a halo, and the weight gradients hand
the tiles to a fixed number of blocks that keep their sums: images smaller than a
tile, one pixel beyond a tile, and a batch with more tiles than three blocks per SM
(36 x 16 = 576 of 152 SMs), each against the FP64 evaluation of the network as
defined (BF16 weights, hidden pre-activations kept in BF16).

Tolerance 5e-3 per tensor: a pre-activation whose FP32 and FP64 sums round to
neighbouring BF16 values is off by 2^-8 = 3.9e-3 at most, and the FP32 backward
signal enters the products with 16 bits (2^-17).
"""
import numpy as np
import pytest

from oracle import cnn as ocnn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402


def _bf16(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()


@pytest.mark.parametrize("n,batch", [(1, 1), (5, 2), (15, 1), (17, 2), (33, 1), (96, 16)])
def test_ragged_and_many_tiles(n, batch):
    params = [(_bf16(w), b) for w, b in ocnn.init_params(5)]
    rng = np.random.default_rng(n)
    params = [(w, b + np.float32(0.1) * rng.standard_normal(b.shape).astype(np.float32)) for w, b in params]
    net = mgdarcy.CNN(n, max_batch=batch, seed=3)
    net.set_params(np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in params]).astype(np.float32))
    x, t = rng.standard_normal((2, batch, 3, n, n)).astype(np.float32)
    xd, td = torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda")
    out = torch.zeros_like(xd)
    net.forward(xd, batch, out)
    loss, g = net.gradients(xd, td, batch)
    y = out.cpu().numpy()
    ref, loss_ref = 0.0, 0.0
    for k in range(batch):
        yr, _ = ocnn.forward(params, x[k].astype(np.float64), _bf16)
        assert np.linalg.norm(y[k] - yr) <= 5e-3 * np.linalg.norm(yr)
        lk, gk = ocnn.loss_and_grads(params, x[k].astype(np.float64), t[k].astype(np.float64), _bf16)
        loss_ref += lk / batch
        ref = ref + np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in gk]) / batch
    assert abs(loss - loss_ref) <= 5e-3 * loss_ref
    k = 0
    for w, b in params:
        for size in (w.size, b.size):
            assert np.linalg.norm(g[k:k + size] - ref[k:k + size]) <= 5e-3 * np.linalg.norm(ref[k:k + size]) + 1e-12
            k += size
    assert k == g.size
