"""Inference on inputs that are infinite, beyond BF16's range or NaN: an infinite
pre-activation saturates the hidden layer (tanh = +-1) and the outputs stay finite,
whatever padding the width needs; a NaN stays in its own row.  Exactly: a finite
1e30 saturates the same units, so its row has the same outputs bit for bit."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,depth", [(40, 2), (33, 1), (250, 3), (1, 2), (256, 2), (64, 1)])
def test_rows_with_infinities_and_nans(width, depth):
    n_in, n_out, rows = 5, 8, 140
    rng = np.random.default_rng(width)
    dims = [n_in] + [width] * depth + [n_out]
    theta = np.concatenate([p for a, b in zip(dims[:-1], dims[1:])
                            for p in (rng.uniform(0.1, 1, a * b) * rng.choice([-1, 1], a * b),
                                      rng.uniform(-0.1, 0.1, b))]).astype(np.float32)
    x = rng.uniform(-1, 1, (rows, n_in)).astype(np.float32)
    m = lbm.lbm_mlp_create(n_in, width, depth, n_out, rows, torch.cuda.current_stream().cuda_stream)
    got = []
    try:
        lbm.lbm_mlp_set_params(m, theta)
        for inf, nan in ((1e30, 0.0), (np.inf, np.nan)):
            x[3, 1], x[64, 0], x[130, 4], x[7, 2] = inf, -inf, min(inf, 3.4e38), nan
            y = torch.empty((rows, n_out), device="cuda")
            lbm.lbm_mlp_forward(m, torch.from_numpy(x).cuda(), rows, y)
            got.append(y.cpu().numpy())
    finally:
        lbm.lbm_mlp_destroy(m)
    assert np.isfinite(got[0]).all() and np.isnan(got[1][7]).all()
    for y in got:
        y[7] = 0.0
    assert np.array_equal(got[0], got[1])
