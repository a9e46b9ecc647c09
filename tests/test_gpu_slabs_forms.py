"""Slabs of a lattice on the other side of a form's size line: a lattice that
marches whose slabs are small enough for the box form, and one in the larger box
whose slabs are small enough for the smaller.  With walls in z the slabs step
exactly as the undivided lattice (the same kernel instantiation); periodic in z
within FP32 rounding, as in every such lattice."""
import numpy as np
import pytest
import torch

from paper_1904_03618_gb300 import lbm, slabs, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny,nz,wall,world,form", [
    (64, 48, 36, (0, 0, 1), 2, 0), (64, 48, 36, (0, 0, 0), 2, 0),   # 110,592 cells, seam form
    (64, 48, 61, (1, 0, 1), 3, 0),                                  # 187,392, tensor copies
    (63, 49, 61, (0, 0, 1), 2, 0),                                  # 188,307, hold form
    (24, 24, 30, (0, 0, 1), 2, 2), (24, 24, 30, (1, 1, 1), 3, 2),   # 17,280: 8 x 4 x 4 boxes
    (80, 40, 40, (0, 0, 1), 3, 0),                                  # whole and slabs march
])
def test_slabs_run_the_form_of_the_undivided_lattice(nx, ny, nz, wall, world, form, storage):
    pd = dict(nx=nx, ny=ny, nz=nz, wall=wall, improved=True, rho_in_R=3.0, rho_in_B=1.0,
              alpha_R=0.9, alpha_B=0.7, tau_R=0.9, tau_B=1.1, A_R=0.001, A_B=0.001, beta=0.7,
              force=(1e-5, 0.0, 0.0))
    refs = (0.0, 0.0 if storage == "f32" else 1.0)
    fields = tuple(np.ascontiguousarray(a, dtype=np.float32)
                   for a in wl.droplet(nx, ny, nz, 0.3 * min(nx, ny, nz), 3.0, 1.0,
                                       velocity=(0.02, 0.01, 0.03), noise=1e-3))
    p = lbm.make_params(storage=storage, **pd)
    p.ref_R, p.ref_B = refs
    whole = lbm.Lattice(p, device=DEV)
    s = slabs.SlabsOnOneDevice(pd, world, device=DEV, storage=storage, refs=refs)
    try:
        assert [lbm.lbm_get_box(x.ctx) for x in [whole] + s.lats] == [form] * (world + 1)
        whole.init_fields(*fields)
        s.init_fields(fields)
        whole.step(8)
        s.step(8)
        for g, r in zip(s.moments(), whole.moments()):
            if wall[2]:
                assert torch.equal(g, r)
            else:
                err = (g.double() - r.double()).abs().max() / r.double().abs().max()
                assert err.item() <= (1e-5 if storage == "f32" else 8 * 2.0 ** -10)
    finally:
        whole.close()
        s.close()
