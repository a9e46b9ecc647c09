"""The box form of the step, the default on small single lattices: against the
marching kernel (an explicitly set configuration) on lattices at its edges --
one cell, extents below, at and just past the 4 x 4 x 4 and 8 x 4 x 4 boxes,
the largest lattices of its range -- with walls, the contact-angle rule,
forces, BGK and 16-bit storage.

Both compute the same step with the same inlined arithmetic; only the
contraction of multiply-add pairs may differ, a few ulp of the largest
population per step: 1e-6 after three steps.  A 16-bit store may then round
the other way: one storage ulp per step."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")

BASE = dict(rho_in_R=3.0, rho_in_B=1.0, alpha_R=0.9, alpha_B=0.7, tau_R=0.8, tau_B=1.1,
            A_R=0.01, A_B=0.01)
CASES = [
    (1, 1, 1, {}), (3, 5, 2, {}), (4, 4, 4, {}), (5, 4, 9, dict(wall=(1, 1, 1))),
    (4, 128, 4, dict(wall=(0, 1, 0), force=(1e-5, 0.0, 0.0))),
    (16, 32, 32, {}),                                                 # 16,384: the last 4^3 box
    (17, 31, 33, dict(wall=(1, 0, 1), wetting=True, contact_angle_deg=60.0)),
    (33, 25, 40, dict(collision="bgk", wall=(0, 0, 1), gravity=(0.0, 0.0, -1e-4))),
    (40, 32, 64, {}),                                                 # 81,920: the last seam lattice
    (33, 31, 29, dict(storage="f16", ref_B=1.0)),
    (40, 30, 21, dict(storage="bf16", ref_B=1.0, wall=(0, 1, 1))),
    (57, 56, 56, {}),                                                 # 178,752, no seam form
]


@pytest.mark.parametrize("nx,ny,nz,kw", CASES)
def test_box_equals_the_marching_kernel(nx, ny, nz, kw):
    p = lbm.make_params(nx, ny, nz, **dict(BASE, **kw))
    fields = wl.random_fields(nx, ny, nz, seed=nx + ny + nz)
    out = []
    for marching in (False, True):
        lat = lbm.Lattice(p, device=DEV, stream=torch.cuda.Stream(DEV))
        try:
            if marching:
                tile_y, zchunk, hold = lbm.lbm_get_fused_config(lat.ctx)
                lbm.lbm_set_fused_config(lat.ctx, 8, 2 if zchunk != 2 else 3, 2)
            lat.init_fields(*fields)
            lat.step(3)
            out.append(lat.get_f().double().cpu().numpy())
        finally:
            lat.close()
    tol = {"f32": 1e-6, "f16": 3 * 2.0 ** -10, "bf16": 3 * 2.0 ** -7}[kw.get("storage", "f32")]
    assert np.abs(out[0] - out[1]).max() <= tol * np.abs(out[1]).max()


def test_graph_of_box_steps_equals_single_steps():
    """Runs of 16 steps replay a captured graph; every length gives the state of single steps."""
    nx, ny, nz = 20, 12, 9
    p = lbm.make_params(nx, ny, nz, wall=(0, 0, 1), **BASE)
    fields = wl.droplet(nx, ny, nz, 3.0, 3.0, 1.0, velocity=(0.02, 0.0, 0.0))
    a = lbm.Lattice(p, device=DEV, stream=torch.cuda.Stream(DEV))
    b = lbm.Lattice(p, device=DEV, stream=torch.cuda.Stream(DEV))
    try:
        a.init_fields(*fields)
        b.init_fields(*fields)
        for n in (35, 1, 20, 50):
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert torch.equal(a.get_f(), b.get_f()), n
        assert a.diagnostics()[12] == 106
    finally:
        a.close()
        b.close()
