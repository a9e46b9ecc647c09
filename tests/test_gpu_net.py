"""The surrogate's whole-network kernels at the edges of their tiles: widths
around the 32-column blocks and their padding, 1 to 8 CTAs of a cluster, rows
around the 32-, 64- and 128-row tiles, more layers than weight buffers, no
hidden layer -- against the FP64 network, at the bars of the layer kernels'
test (BF16 operands: relative rounding 2^-9 through a few layers); the largest
batch of the three-kernel training step against the layer-by-layer path; and
outputs in host memory, on top of the inputs, and past one round of tiles."""
import numpy as np
import pytest
import torch

from oracle import mlp as ref
from paper_1904_03618_gb300 import lbm

pytestmark = pytest.mark.gpu


def _theta(rng, dims):
    parts = []
    for a, b in zip(dims[:-1], dims[1:]):
        parts += [rng.uniform(-1, 1, a * b) * np.sqrt(6.0 / (a + b)), rng.uniform(-0.1, 0.1, b)]
    return np.concatenate(parts).astype(np.float32)


def _net(n_in, width, depth, n_out, batch, seed=3):
    rng = np.random.default_rng(seed)
    theta = _theta(rng, [n_in] + [width] * depth + [n_out])
    m = lbm.lbm_mlp_create(n_in, width, depth, n_out, batch, torch.cuda.current_stream().cuda_stream)
    lbm.lbm_mlp_set_params(m, theta)
    x = torch.from_numpy(rng.uniform(-1, 1, (batch, n_in)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(-1, 1, (batch, n_out)).astype(np.float32)).cuda()
    return m, theta, x, t


@pytest.mark.parametrize("n_in,width,depth,n_out,batch", [
    (1, 1, 1, 1, 1), (5, 31, 2, 33, 31), (5, 32, 1, 8, 32), (33, 65, 2, 16, 33), (5, 96, 3, 7, 127),
    (5, 200, 3, 16, 128), (5, 256, 4, 16, 129), (3, 256, 6, 256, 257), (256, 40, 0, 100, 65),
    (5, 250, 2, 16, 1000),
])
def test_forward_loss_and_gradient(n_in, width, depth, n_out, batch):
    m, theta, x, t = _net(n_in, width, depth, n_out, batch)
    try:
        y = torch.full((batch, n_out), float("nan"), device="cuda")
        lbm.lbm_mlp_forward(m, x, batch, y)
        g = np.full(theta.size, np.nan, dtype=np.float32)
        loss = lbm.lbm_mlp_loss_grad(m, x, t, batch, g)
    finally:
        lbm.lbm_mlp_destroy(m)
    th, xx, tt = (v.astype(np.float64) for v in (theta, x.cpu().numpy(), t.cpu().numpy()))
    y_ref, _ = ref.forward(th, xx, n_in, width, depth, n_out)
    loss_ref, g_ref = ref.loss_and_grad(th, xx, tt, n_in, width, depth, n_out)
    scale = np.sqrt(np.mean(y_ref ** 2)) + 1e-12
    assert np.max(np.abs(y.cpu().numpy() - y_ref)) <= 2e-2 * scale
    assert abs(loss - loss_ref) <= 2e-2 * loss_ref
    for (gw, gb), (rw, rb) in zip(ref.unpack(g.astype(np.float64), n_in, width, depth, n_out),
                                  ref.unpack(g_ref, n_in, width, depth, n_out)):
        for a, b in ((gw, rw), (gb, rb)):
            assert np.linalg.norm(a - b) <= 3e-2 * np.linalg.norm(g_ref) + 1e-7


def test_largest_fused_batches_equal_the_layer_path():
    """2 x 2080 rows through the three-kernel path average to 4160 rows through
    the layer-by-layer one: the operands round alike (the loss scales differ by
    a power of two), only FP32 sums differ in order -- K = 4160 terms, at most
    4160 * 2^-24 = 2.5e-4 of sum |a b|, in the norm far less: 1e-5."""
    dims = (5, 256, 3, 16)
    m, theta, x, t = _net(*dims, 4160)
    try:
        whole, half = np.empty(theta.size, np.float32), np.zeros(theta.size, np.float64)
        loss = lbm.lbm_mlp_loss_grad(m, x, t, 4160, whole)
        parts = []
        for k in (0, 1):
            g = np.empty(theta.size, np.float32)
            parts.append(lbm.lbm_mlp_loss_grad(m, x[k * 2080:(k + 1) * 2080].contiguous(),
                                               t[k * 2080:(k + 1) * 2080].contiguous(), 2080, g))
            half += 0.5 * g
    finally:
        lbm.lbm_mlp_destroy(m)
    assert abs(loss - 0.5 * sum(parts)) <= 1e-5 * loss
    assert np.linalg.norm(whole - half) <= 1e-5 * np.linalg.norm(half)


def test_outputs_in_host_memory_over_the_inputs_and_past_one_round():
    rows = 152 * 128 * 2 + 77  # three tiles on some CTAs, a ragged last one
    m, theta, x, _ = _net(6, 64, 2, 6, rows)
    try:
        y = torch.empty((rows, 6), device="cuda")
        lbm.lbm_mlp_forward(m, x, rows, y)
        host = np.empty((rows, 6), np.float32)
        lbm.lbm_mlp_forward(m, x, rows, host)
        part = torch.empty((100, 6), device="cuda")
        lbm.lbm_mlp_forward(m, x[rows - 100:].contiguous(), 100, part)
        lbm.lbm_mlp_forward(m, x, rows, x)  # in place
        assert np.array_equal(host, y.cpu().numpy())
        assert torch.equal(part, y[rows - 100:]) and torch.equal(x, y)
    finally:
        lbm.lbm_mlp_destroy(m)
