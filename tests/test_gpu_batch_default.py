"""The form a batch runs by default follows its boxes' tiles: batches on either
side of each line pick the form the schedule estimates name, and step as under
the 34 x 15 tensor-copy form (the same arithmetic; the contraction of
multiply-add pairs may differ, a few ulp of the largest population per step:
1e-6 after three steps, one storage ulp per step in 16 bits)."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
BASE = dict(rho_in_R=3.0, alpha_R=0.9, alpha_B=0.7, tau_R=0.8, tau_B=1.1, A_R=0.01, A_B=0.01,
            wall=(0, 0, 1), ref_B=1.0)


@pytest.mark.parametrize("box,n,storage,want", [
    ((40, 40, 24), 3, "f32", (15, 32, 8)),      # 24 CTAs: too few to choose
    ((40, 40, 24), 4, "f32", (8, 12, 2)),       # 32
    ((64, 64, 32), 32, "f32", (12, 32, 7)),     # every tile on both seams' rows and columns
    ((96, 64, 24), 20, "f32", (15, 32, 8)),
    ((32, 64, 32), 40, "f32", (15, 32, 8)),     # narrower than the seam form's tile
    ((40, 40, 24), 20, "f16", (8, 12, 2)),
    ((96, 64, 32), 8, "bf16", (15, 32, 7)),
])
def test_default_form_of_a_batch(box, n, storage, want):
    nx, ny, nz = box
    ps = [lbm.make_params(nx, ny, nz, storage=storage, **BASE) for _ in range(n)]
    got = []
    for explicit in (False, True):
        b = lbm.Batch(ps, device=DEV, stream=torch.cuda.Stream(DEV))
        try:
            if explicit:
                lbm.lbm_set_fused_config(b.ctx, 15, 32, 8 if storage == "f32" else 7)
            else:
                assert lbm.lbm_get_fused_config(b.ctx) == want
            for k in range(n):
                b.init_fields(k, *wl.droplet(nx, ny, nz, 6.0, 3.0, 1.0, velocity=(0.02, 0.01, 0.0),
                                             noise=1e-2, seed=k))
            b.step(3)
            got.append([b.get_f(k).double().cpu().numpy() for k in (0, n - 1)])
        finally:
            b.close()
    tol = {"f32": 1e-6, "f16": 3 * 2.0 ** -10, "bf16": 3 * 2.0 ** -7}[storage]
    for a, r in zip(*got):
        assert np.abs(a - r).max() <= tol * np.abs(r).max()
