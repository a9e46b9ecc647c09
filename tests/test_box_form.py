"""Which kernel steps a small lattice: lbm_default_box on both sides of each of
its lines (host only), and on the GPU that a context runs the form it reports --
that a configuration set explicitly runs the kernel it names, also when it is the
one lbm_create reports: the tensor-copy kernels are the ones whose stage waits
give up under a 1 ns limit (bounded waits: the kernel drains its copies and
returns)."""
import ctypes

import pytest

from paper_1904_03618_gb300 import lbm, workloads as wl


@pytest.mark.parametrize("shape,kw,want", [
    ((1, 1, 1), {}, 1), ((16, 32, 32), {}, 1), ((16, 32, 33), {}, 2),
    ((40, 32, 64), {}, 2), ((40, 32, 65), {}, 0),                       # seam lattices: 81,920
    ((40, 32, 65), dict(wall=(1, 0, 0)), 2), ((41, 32, 65), {}, 2),     # no seam form
    ((32, 32, 81), {}, 2),                                              # narrower than the seam tile
    ((40, 32, 65), dict(storage="f16"), 0), ((42, 32, 65), dict(storage="f16"), 2),
    ((100, 36, 50), dict(wall=(0, 1, 0)), 2), ((100, 36, 51), dict(wall=(0, 1, 0)), 0),  # 180,000
    ((16, 16, 16), dict(collision="bgk"), 0), ((16, 16, 16), dict(kernel="two_pass"), 0),
    ((4000, 4000, 4000), {}, 0),                                        # too large for one context
])
def test_default_box(shape, kw, want):
    assert lbm.lbm_default_box(lbm.make_params(*shape, **kw)) == want


def test_default_box_refuses_what_create_refuses():
    with pytest.raises(lbm.LbmError):
        lbm.lbm_default_box(lbm.make_params(16, 16, 16, tau_R=0.2))
    assert lbm._lib.lbm_default_box(ctypes.byref(lbm.make_params(4, 4, 4)), None) == lbm.LBM_ERR_ARG
    assert lbm._lib.lbm_set_box(None, 1) == lbm.LBM_ERR_ARG and lbm._lib.lbm_get_box(None) == 0


BASE = dict(rho_in_R=3.0, rho_in_B=1.0, alpha_R=0.9, alpha_B=0.7, tau_R=0.8, tau_B=1.1,
            A_R=0.01, A_B=0.01)


def _lattice(shape, **kw):
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda:0")
    ref_B = kw.pop("ref_B", 0.0)
    p = lbm.make_params(*shape, **dict(BASE, **kw))
    p.ref_B = ref_B
    lat = lbm.Lattice(p, device=dev, stream=torch.cuda.Stream(dev))
    lat.init_fields(*wl.droplet(*shape, 0.3 * min(shape), 3.0, 1.0, velocity=(0.02, 0.01, 0.0),
                                noise=1e-3))
    return p, lat


def _waits_for_copies(lat, steps=6):
    """Whether a step under the 1 ns limit of the stage waits reports a give-up."""
    L = lbm._lib
    L.lbm_test_set_wait_limits.argtypes = [ctypes.c_ulonglong, ctypes.c_ulonglong]
    out = (ctypes.c_double * 16)()
    assert L.lbm_test_set_wait_limits(1, 0) == lbm.LBM_OK
    try:
        for _ in range(steps):
            lbm.lbm_step(lat.ctx, 1)
            if L.lbm_diagnostics(lat.ctx, out) == lbm.LBM_ERR_TIMEOUT:
                return True
    finally:
        assert L.lbm_test_set_wait_limits(0, 0) == lbm.LBM_OK
    return False


@pytest.mark.gpu
@pytest.mark.parametrize("shape,kw", [
    ((64, 24, 16), {}), ((34, 15, 6), dict(wall=(0, 0, 1))),
    ((64, 24, 16), dict(storage="f16", ref_B=1.0)), ((68, 30, 9), dict(storage="bf16", ref_B=1.0)),
    ((64, 24, 16), dict(wall=(1, 1, 0))),
])
def test_the_reported_configuration_runs_its_kernel_when_set(shape, kw):
    p, lat = _lattice(shape, **kw)
    try:
        assert lbm.lbm_get_box(lat.ctx) == lbm.lbm_default_box(p) > 0
        assert not _waits_for_copies(lat)          # the box form has none
        config = lbm.lbm_get_fused_config(lat.ctx)
        lbm.lbm_set_fused_config(lat.ctx, *config)
        assert lbm.lbm_get_box(lat.ctx) == 0 and lbm.lbm_get_fused_config(lat.ctx) == config
        assert _waits_for_copies(lat) == (config[2] in (7, 8))
        if shape[:2] == (64, 24):
            assert config[2] in (7, 8)             # the tensor-copy kernels are among them
    finally:
        lat.close()


@pytest.mark.gpu
def test_choosing_the_form():
    torch = pytest.importorskip("torch")
    fields = wl.droplet(24, 20, 16, 5.0, 3.0, 1.0, velocity=(0.02, 0.01, 0.0), noise=1e-3)
    p, lat = _lattice((24, 20, 16))
    ref = _lattice((24, 20, 16))[1]
    try:
        ref.init_fields(*fields)
        ref.step(5)
        # away from the default and back (graphs captured in between): the same steps
        lbm.lbm_set_fused_config(lat.ctx, 8, 4, 2)
        lat.step(24)
        lbm.lbm_set_box(lat.ctx, 2)
        assert lbm.lbm_get_box(lat.ctx) == 2
        lat.step(24)
        lbm.lbm_set_box(lat.ctx, lbm.lbm_default_box(p))
        lat.init_fields(*fields)
        lat.step(5)
        assert torch.equal(lat.get_f(), ref.get_f())
        for bad in (-1, 3):
            with pytest.raises(lbm.LbmError):
                lbm.lbm_set_box(lat.ctx, bad)
    finally:
        lat.close()
        ref.close()
    for kw in (dict(collision="bgk"), dict(kernel="two_pass")):
        p, lat = _lattice((24, 20, 16), **kw)
        try:
            assert lbm.lbm_get_box(lat.ctx) == 0
            lbm.lbm_set_box(lat.ctx, 0)
            with pytest.raises(lbm.LbmError):
                lbm.lbm_set_box(lat.ctx, 1)
        finally:
            lat.close()
    b = lbm.Batch([lbm.make_params(8, 8, 8, **BASE)] * 2, device=torch.device("cuda:0"))
    try:
        with pytest.raises(lbm.LbmError):
            lbm.lbm_set_box(b.ctx, 1)
    finally:
        b.close()
