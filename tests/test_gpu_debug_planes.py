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
