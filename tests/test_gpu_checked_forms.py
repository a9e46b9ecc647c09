"""The index-checked build over every form of the step, named one by one: the
default configurations of lattices this small run the box form, so the marching
forms -- tensor-copy, seam, hold -- are set explicitly here.  No index out of
range over a few steps, and the populations of the normal build."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PERIODIC, ZWALL, XYWALL = (0, 0, 0), (0, 0, 1), (1, 1, 0)
# (nx, ny, nz, wall, storage, (tile_y, zchunk, hold) or box form)
CASES = [
    (67, 23, 11, wall, st, (ty, zc, hold))
    for wall in (PERIODIC, (1, 1, 1)) for st in ("f32", "f16")
    for ty, zc, hold in ((8, 0, 0), (8, 3, 1), (8, 4, 2), (8, 0, 3), (16, 5, 4), (8, 3, 5),
                         (8, 0, 6), (16, 4, 0), (16, 0, 1))
] + [
    (68, 23, 11, wall, st, (ty, zc, hold))
    for wall in (XYWALL, (1, 0, 1)) for st in ("f32", "f16", "bf16")
    for ty, zc, hold in ((8, 0, 7), (8, 4, 8), (15, 3, 7), (15, 0, 8))
] + [
    (nx, ny, nz, wall, st, (ty, 0, hold))
    for nx, ny, nz in ((34, 15, 6), (68, 30, 9), (100, 23, 11))
    for wall in (PERIODIC, ZWALL)
    for st, ty, hold in (("f32", 12, 7), ("f32", 15, 8), ("f32", 15, 7), ("f16", 12, 7),
                         ("f16", 15, 7), ("bf16", 15, 7))
    if st == "f32" or nx % 4 == 0
] + [
    (13, 9, 5, wall, st, box) for wall in (PERIODIC, ZWALL, (1, 1, 1)) for st in ("f32", "f16")
    for box in (1, 2)
]

SCRIPT = r"""
import ctypes, json, sys
import numpy as np
import torch
from paper_1904_03618_gb300 import lbm, workloads as wl

dev = torch.device("cuda:0")
counts = []
for k, (nx, ny, nz, wall, st, form) in enumerate(json.loads(sys.argv[1])):
    p = lbm.make_params(nx, ny, nz, wall=tuple(wall), storage=st, rho_in_R=3.0, rho_in_B=1.0,
                        alpha_R=0.9, alpha_B=0.7, tau_R=0.8, tau_B=1.1, A_R=0.01, A_B=0.01,
                        force=(2e-5, 0.0, 0.0), wetting=bool(wall[2]), contact_angle_deg=60.0)
    p.ref_B = 0.0 if st == "f32" else 1.0
    lat = lbm.Lattice(p, device=dev)
    if isinstance(form, list):
        lbm.lbm_set_fused_config(lat.ctx, *form)
        assert lbm.lbm_get_box(lat.ctx) == 0
    else:
        lbm.lbm_set_box(lat.ctx, form)
    lat.init_fields(*wl.random_fields(nx, ny, nz, seed=k))
    lat.step(3)
    np.save("%s/%d.npy" % (sys.argv[2], k), lat.get_f().cpu().numpy())
    c, n = ctypes.c_int(), ctypes.c_uint()
    assert lbm._lib.lbm_test_index_checks(lat.ctx, ctypes.byref(c), ctypes.byref(n)) == 0
    counts.append([c.value, n.value])
    lat.close()
print(json.dumps(counts))
"""


def _run(lib, outdir):
    outdir.mkdir()
    r = subprocess.run([sys.executable, "-c", SCRIPT, json.dumps(CASES), str(outdir)],
                       env=dict(os.environ, LBM_LIBRARY=lib), cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_every_form_counts_no_index_out_of_range(tmp_path):
    import __graft_entry__ as g
    got = _run(g.build_checked(), tmp_path / "c")
    ref = _run(os.path.join(ROOT, "paper_1904_03618_gb300", "_lib", "liblbm.so"), tmp_path / "n")
    for k, case in enumerate(CASES):
        assert got[k] == [1, 0], (case, got[k])  # checked build, nothing out of range
        assert ref[k] == [0, 0], (case, ref[k])
        a, b = (np.load(tmp_path / d / ("%d.npy" % k)) for d in "cn")
        assert np.all(np.isfinite(a)), case
        # the same arithmetic; where another multiply-add pair is contracted a
        # 16-bit store can round the other way: one storage ulp
        tol = {"f32": 1e-6, "f16": 2.0 ** -10, "bf16": 2.0 ** -7}[case[4]]
        assert np.abs(a - b).max() <= tol * max(np.abs(b).max(), 1.0), case
