"""The index-checking build on the fused y/z pass and the far field's inverse y pass: their checks pass, over planes with
paired and single loads, rows and columns that do not fill a warp and several rounds per warp, and a probe that takes
the last element they store as out of range shows that they are made.  Runs in a child process (the debug library is
chosen at import)."""
import os
import subprocess
import sys

import pytest

from gpu_common import torch_and_lib

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PREAMBLE = r'''
import os, sys
import numpy as np
import torch
import paper_1910_13844_gb300 as ls
import phantoms as ph
from gpu_common import ETA_B, H, KB, LAM, potential, rel, to_dev
from oracle import model
assert ls.library_path().endswith("libls_debug.so"), ls.library_path()

def site():
    checked, s = ls.ls_debug_bounds(clear=True)
    assert checked
    return s

assert site() == 0
'''

CHILD = PREAMBLE + r'''
for shape in [(8, 8, 16), (24, 48, 16), (16, 12, 24), (72, 72, 16), (96, 128, 16), (144, 144, 16), (12, 144, 16), (96, 192, 16)]:
    f64 = potential(ph.random_potential_like(shape, seed=3))
    f = to_dev(torch, f64, torch.float32)
    f64 = f.cpu().numpy().astype(np.float64)
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    plan = ls.Plan(shape, KB, H)
    x = torch.stack([to_dev(torch, ph.random_field(shape, q), torch.complex64) for q in range(2)])
    r = torch.stack([to_dev(torch, ph.random_field(shape[1:], 9 + q), torch.complex64) for q in range(2)])
    y, far, back = torch.empty_like(x), plan.detector(2), plan.field(2)
    for adjoint in (False, True):
        ls.ls_matvec_batch(plan.handle, f, x, y, adjoint)
        torch.cuda.synchronize()
        assert site() == 0, shape
        for q in range(2):
            assert rel(y[q].cpu().numpy(), op.A(x[q].cpu().numpy().astype(np.complex128), f64, adjoint)) < 3e-6
    ls.ls_farfield(plan.handle, f, x, far)
    ls.ls_farfield_adjoint(plan.handle, r, back)
    assert site() == 0, shape
    for q in range(2):
        assert rel(far[q].cpu().numpy(), op.farfield_fft(f64 * x[q].cpu().numpy().astype(np.complex128))) < 3e-6
        assert rel(back[q].cpu().numpy(), op.farfield_adjoint_fft(r[q].cpu().numpy().astype(np.complex128))) < 3e-6
    # probes: a failed check is recorded and its access skipped
    ls.ls_debug_inject(plan.handle, ls.LS_INJECT_BOUNDS_PROBE, 2)
    ls.ls_matvec_batch(plan.handle, f, x, y)
    torch.cuda.synchronize()
    assert site() == 0x701, shape
    ls.ls_debug_inject(plan.handle, ls.LS_INJECT_BOUNDS_PROBE, 3)
    ls.ls_farfield(plan.handle, f, x, far)
    assert site() == 0x803, shape
    ls.ls_farfield_adjoint(plan.handle, r, back)
    assert site() == 0x803, shape
    ls.ls_debug_inject(plan.handle, ls.LS_INJECT_NONE, 0)
    ls.ls_matvec_batch(plan.handle, f, x, y)
    torch.cuda.synchronize()
    assert site() == 0, shape
    plan.close()
    print(shape, "ok", flush=True)
print("all ok", flush=True)
'''


def run_debug_child(code, **env):
    torch_and_lib()
    import __graft_entry__

    __graft_entry__._build_module().build(debug=True)
    env = dict(os.environ, LS_DEBUG_BOUNDS="1", **env)
    env["PYTHONPATH"] = ROOT + os.pathsep + HERE + os.pathsep + env.get("PYTHONPATH", "")
    r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0 and "all ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


@pytest.mark.gpu
def test_checks_pass_and_are_made():
    run_debug_child(CHILD)


FORMS = PREAMBLE + r'''
name = torch.cuda.get_device_name().replace(" ", "_")

def case(shape, views, line):
    nz, ny, nx = shape
    open(os.environ["LS_AUTOTUNE_CACHE"], "w").write(f"{name}:{nx}x{ny}x{nz}:{views} {line}\n")
    f64 = potential(ph.random_ellipsoids(shape, count=3, rmin=2, rmax=6, dn_max=0.04, seed=3))
    f = to_dev(torch, f64, torch.float32)
    kvec = ph.cone_directions(views, 0.8) * KB
    plan = ls.Plan(shape, KB, H, tol=1e-6)
    assert plan.autotune(views, f)["from_cache"] == 1
    u, far, code, stats = plan.forward(f, plan.plane_waves(kvec))
    g, gcode, _ = plan.gradient(f, far.clone(), u_fwd=u)
    torch.cuda.synchronize()
    assert code == ls.LS_OK and gcode == ls.LS_OK, (shape, line, stats)
    assert site() == 0, (shape, line)
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    for q in range(views):
        u_o = model.forward(op, f64, model.plane_wave(shape, H, kvec[q]), tol=1e-12)
        assert rel(u[q].cpu().numpy(), u_o) < 1e-4, (shape, line)
        assert rel(far[q].cpu().numpy(), op.farfield_fft(f64 * u_o)) < 1e-4, (shape, line)
    assert bool(torch.isfinite(g).all())
    plan.close()

# z_tma ix_prefetch fx_views_fastest check_every use_graphs ms ms z_split strided_wide views_per_launch z_persist fx_bulk fused
# the three passes at the lengths whose z pass has a kernel or a split of its own (144: column groups; 128, 192 and 384:
# several stage-2 sub-transforms per thread), in every form, and at one that does not
for shape in [(72, 16, 16), (64, 16, 16), (96, 16, 16), (192, 16, 16), (24, 16, 32)]:
    for form in ["1 1 0 2 1 1 1 0 0 0 0 0 0", "1 0 1 2 0 1 1 1 1 1 1 0 0", "1 1 0 4 1 1 1 0 1 0 2 1 0", "0 1 0 2 1 1 1 0 0 0 0 0 0"]:
        case(shape, 2, form)
    print(shape, "ok", flush=True)
# the fused pass beside every form of the first and last pass
for form in ["1 1 1 2 1 1 1 0 0 0 0 0 1", "1 0 0 2 1 1 1 0 0 0 0 1 1", "1 1 0 4 0 1 1 0 0 1 0 1 1", "1 0 1 8 1 1 1 0 0 2 0 0 1"]:
    for shape in [(32, 32, 32), (24, 16, 96), (72, 72, 16)]:
        case(shape, 3, form)
print("all ok", flush=True)
'''


@pytest.mark.gpu
def test_every_form_of_a_tuned_plan(tmp_path):
    run_debug_child(FORMS, LS_AUTOTUNE_CACHE=str(tmp_path / "tune.txt"))
