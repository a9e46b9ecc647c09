"""FP32 single lattices without walls in x or y run a collision with fewer
operations in their default forms; the register-hold form (tile_y 8, hold 0)
keeps the first one, and the default forms of a lattice with x or y walls do
too.

The two sum a population from about 20 terms no larger than the largest
population: 20 x 2^-24 = 1.2e-6 of it per step and side, so 1e-5 after three
steps.  With walls in x or y the arithmetic is the same but for the contraction
of multiply-add pairs: 1e-6."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")

BASE = dict(rho_in_R=3.0, rho_in_B=1.0, alpha_R=0.9, alpha_B=0.7, tau_R=0.8, tau_B=1.1,
            A_R=0.01, A_B=0.01, force=(2e-5, 0.0, 0.0), gravity=(0.0, 0.0, -1e-5))
BOX, HOLD2, TMA, SEAM15, SEAM12 = None, (8, 2), (8, 8), (15, 8), (12, 7)
CASES = [
    (7, 5, 3, BOX, {}), (33, 31, 29, BOX, dict(wall=(0, 0, 1))),
    (31, 15, 9, HOLD2, {}), (40, 26, 13, HOLD2, dict(wall=(0, 0, 1))),
    (40, 26, 13, HOLD2, dict(wall=(0, 1, 1))), (33, 20, 9, HOLD2, dict(wall=(1, 0, 0))),
    (64, 23, 14, TMA, dict(wall=(0, 0, 1))), (64, 23, 14, TMA, {}),
    (64, 23, 14, TMA, dict(wall=(1, 0, 1))),
    (72, 37, 19, SEAM15, {}), (72, 37, 19, SEAM15, dict(wall=(0, 0, 1))),
    (72, 37, 19, SEAM12, {}), (72, 37, 19, SEAM12, dict(wall=(0, 0, 1))),
]


@pytest.mark.parametrize("nx,ny,nz,form,kw", CASES)
def test_default_forms_equal_the_register_hold_form(nx, ny, nz, form, kw):
    p = lbm.make_params(nx, ny, nz, **dict(BASE, **kw))
    fields = wl.random_fields(nx, ny, nz, seed=nx + ny + nz)
    out = []
    for tile_hold in (form, (8, 0)):
        lat = lbm.Lattice(p, device=DEV)
        try:
            if tile_hold:
                lbm.lbm_set_fused_config(lat.ctx, tile_hold[0], 3, tile_hold[1])
            lat.init_fields(*fields)
            lat.step(3)
            out.append(lat.get_f().double().cpu().numpy())
        finally:
            lat.close()
    wall = kw.get("wall", (0, 0, 0))
    tol = 1e-6 if wall[0] or wall[1] else 1e-5
    assert np.abs(out[0] - out[1]).max() <= tol * np.abs(out[1]).max()
