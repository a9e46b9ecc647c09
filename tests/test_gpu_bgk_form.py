"""BGK lattices of every size step in the shared-memory-hold kernel: under that
operator (every rate 1 / tau_v) a last bit that another form contracts differently
grows near tau_v = 1/2, so the default is that kernel bit for bit, whatever the
z chunk."""
import pytest
import torch

from paper_1904_03618_gb300 import lbm, rt, workloads as wl

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("nx,ny,nz,wall", [
    (24, 24, 96, (0, 0, 1)), (40, 33, 29, (1, 1, 1)), (4, 128, 4, (0, 1, 0)), (40, 40, 40, (0, 0, 0)),
])
def test_bgk_default_is_the_hold_kernel(nx, ny, nz, wall, storage):
    pd = dict(rt.rt_params(L=24), nx=nx, ny=ny, nz=nz, wall=wall, collision="bgk", storage=storage)
    p = lbm.make_params(**pd)
    p.ref_R, p.ref_B = pd["rho_in_R"], pd["rho_in_B"]
    rR, rB, u = wl.rayleigh_taylor(nx, ny, nz, nx, 0.1, nz // 2, 3.0, 1.0)
    u[2] += 0.02 * (rR - rB) / 3.0
    u[0] += 0.03 * (rB > 0)
    out = []
    for config in (None, (8, 5, 2)):
        lat = lbm.Lattice(p, device=DEV, stream=torch.cuda.Stream(DEV))
        try:
            if config:
                lbm.lbm_set_fused_config(lat.ctx, *config)
            lat.init_fields(rR, rB, u)
            lat.step(24)
            out.append(lat.get_f())
        finally:
            lat.close()
    assert torch.isfinite(out[1]).all()
    assert torch.equal(*out)
