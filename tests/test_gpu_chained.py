"""Kernels launched with programmatic stream serialisation (the box form of the
step, the surrogate's training step) wait on the GPU while the kernel that
writes their input still runs.  Several hundred of them queued back to back,
with grids small enough that two or three fit the GPU at once, give bit for bit
what they give with a synchronisation after each."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,kw", [
    ((24, 24, 24), {}), ((24, 24, 24), dict(storage="f16", ref_B=1.0)),      # 216 boxes
    ((20, 16, 16), dict(wall=(0, 0, 1))), ((4, 128, 4), dict(wall=(0, 1, 0))),  # 80, 32
    ((40, 32, 32), dict(wall=(1, 0, 1))),                                    # 8 x 4 x 4: 320
])
def test_queued_box_steps_equal_synchronised_ones(n, kw):
    p = lbm.make_params(*n, **dict(dict(rho_in_R=3.0, alpha_R=0.9, alpha_B=0.7, tau_R=0.8,
                                        tau_B=1.1, A_R=0.01, A_B=0.01), **kw))
    fields = wl.droplet(*n, 0.3 * min(n), 3.0, 1.0, velocity=(0.03, 0.02, 0.01), noise=1e-2)
    out = []
    for queued in ("graph", "launches", None):
        stream = torch.cuda.Stream(DEV)
        lat = lbm.Lattice(p, device=DEV, stream=stream)
        try:
            lat.init_fields(*fields)
            if queued == "graph":
                lat.step(400)
            else:
                for _ in range(400):
                    lat.step(1)
                    if not queued:
                        stream.synchronize()
            out.append(lat.get_f())
        finally:
            lat.close()
    assert torch.isfinite(out[2]).all()
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[2])


@pytest.mark.parametrize("batch,width,depth", [(32, 64, 1), (256, 256, 4), (200, 96, 3)])
def test_queued_training_steps_equal_synchronised_ones(batch, width, depth):
    # up to 256 rows: no atomics, the sums have one order
    stream = torch.cuda.Stream(DEV)
    out = []
    for queued in (True, False):
        m = lbm.lbm_mlp_create(5, width, depth, 16, batch, stream.cuda_stream)
        try:
            theta = np.random.default_rng(3).uniform(-0.1, 0.1, lbm.lbm_mlp_num_params(m))
            lbm.lbm_mlp_set_params(m, theta.astype(np.float32))
            g = torch.Generator().manual_seed(7)
            xs = (2 * torch.rand((8, batch, 5), generator=g) - 1).cuda()
            ts = (2 * torch.rand((8, batch, 16), generator=g) - 1).cuda()
            torch.cuda.synchronize()
            for k in range(200):
                lbm.lbm_mlp_train_step(m, xs[k % 8], ts[k % 8], batch, 1e-3, want_loss=False)
                if not queued:
                    stream.synchronize()
            got = np.empty(theta.size, np.float32)
            lbm.lbm_mlp_get_params(m, got)
            stream.synchronize()
            out.append(got)
        finally:
            lbm.lbm_mlp_destroy(m)
    assert np.isfinite(out[1]).all() and not np.array_equal(out[1], theta.astype(np.float32))
    assert np.array_equal(out[0], out[1])
