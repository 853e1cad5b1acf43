"""Which form of the y/z passes the launches of a tuned plan run, read from their NVTX ranges: the fused pass opens
the ranges of FY, Z and IY inside one another, the three passes one after the other."""
import pytest

import phantoms as ph
from oracle import model

from gpu_common import ETA_B, H, KB, LAM, potential, rel, to_dev, torch_and_lib
from test_gpu_autotune import VARIANTS
from test_trace import _run

SOLVE = """
    import os
    import numpy as np, torch
    import paper_1910_13844_gb300 as ls
    import phantoms as ph
    from gpu_common import ETA_B, H, KB, LAM, potential, rel, to_dev
    from oracle import model
    shape, views, line = {shape}, {views}, "{line}"
    nz, ny, nx = shape
    name = torch.cuda.get_device_name().replace(" ", "_")
    os.environ["LS_AUTOTUNE_CACHE"] = r"{cache}"
    open(r"{cache}", "w").write(f"{{name}}:{{nx}}x{{ny}}x{{nz}}:{{views}} {{line}}\\n")
    f64 = potential(ph.random_ellipsoids(shape, count=3, rmin=2, rmax=6, dn_max=0.04))
    f = to_dev(torch, f64, torch.float32)
    plan = ls.Plan(shape, KB, H, tol=1e-6)
    k = ph.cone_directions(views, 0.8) * KB
    t = plan.autotune(views, f)
    assert t["from_cache"] == 1
    u, far, code, stats = plan.forward(f, plan.plane_waves(k))
    torch.cuda.synchronize()
    assert code == ls.LS_OK
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    for q in (0, views // 2, views - 1):
        u_o = model.forward(op, f64, model.plane_wave(shape, H, k[q]), tol=1e-12)
        assert rel(u[q].cpu().numpy(), u_o) < 1e-4
    plan.close()
"""


def forms(lines):
    """For every operator application between the solve's start and end: True if its FY, Z and IY are one launch."""
    i = lines.index("push solve")
    out = []
    for a, b in zip(lines[i:], lines[i + 1:]):
        if a == "push FY":
            out.append(b == "push Z")
    return out


def solve_forms(tmp_path, monkeypatch, shape, views, line):
    import os
    monkeypatch.setenv("PYTHONPATH", os.path.dirname(os.path.abspath(__file__)))
    lines = _run(tmp_path, SOLVE.format(shape=shape, views=views, line=line, cache=tmp_path / "tune.txt"))
    # the far field that follows the solve runs FY alone
    n = len(forms(lines)) - 1
    assert n >= 4
    return forms(lines)[:n]


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [0, 1, None])
@pytest.mark.parametrize("chunk", [0, 1, 2])
def test_chunks_of_a_batch_run_the_form_chosen_for_it(tmp_path, monkeypatch, chunk, fused):
    torch_and_lib()
    line = f"1 1 0 2 0 1.0 1.0 0 0 {chunk} 0 0" + ("" if fused is None else f" {fused}")
    assert set(solve_forms(tmp_path, monkeypatch, (32, 32, 32), 3, line)) == {bool(fused)}


@pytest.mark.gpu
def test_chunks_of_a_pair_that_is_fused_only_by_choice(tmp_path, monkeypatch):
    # nz = 8: by default the three passes in launches of more than two waves of CTAs
    torch_and_lib()
    line = "1 1 0 2 0 1.0 1.0 0 0 40 0 0 1"
    assert set(solve_forms(tmp_path, monkeypatch, (8, 32, 64), 80, line)) == {True}


@pytest.mark.gpu
def test_the_tuner_tries_the_first_and_last_pass_in_both_forms(tmp_path):
    # before its first solve: the prefetch and the grid order, two values each, in the three passes and the fused one
    torch_and_lib()
    lines = _run(tmp_path, """
        import torch
        import paper_1910_13844_gb300 as ls
        plan = ls.Plan((16, 16, 16), 8.0, 0.1)
        t = plan.autotune(2, torch.full((16, 16, 16), 0.5, device="cuda"))
        assert t["from_cache"] == 0
        plan.close()
    """)
    before = lines[:lines.index("push solve")]
    runs = [b == "push Z" for a, b in zip(before, before[1:]) if a == "push FY"]
    per_variant = 1 + 4   # one compared, one untimed and three timed
    assert runs.count(True) == 4 * per_variant
    assert runs.count(False) >= 4 * per_variant


@pytest.mark.gpu
@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("variant", VARIANTS)
def test_every_variant_in_both_forms(tmp_path, monkeypatch, variant, fused):
    # SOLVE compares the fields with the oracle's
    torch_and_lib()
    v = [str(x) for x in variant]
    line = " ".join(v[:5]) + " 1.0 1.0 " + " ".join(v[5:]) + f" {fused}"
    assert set(solve_forms(tmp_path, monkeypatch, (32, 32, 32), 3, line)) == {bool(fused)}


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(72, 72, 16), (144, 144, 16), (8, 64, 32), (48, 8, 96)])
def test_several_planes_per_cta_where_the_fused_pass_is_a_choice(tmp_path, monkeypatch, shape):
    torch, ls = torch_and_lib()
    views, (nz, ny, nx) = 70, shape
    cache = tmp_path / "tune.txt"
    name = torch.cuda.get_device_name().replace(" ", "_")
    cache.write_text(f"{name}:{nx}x{ny}x{nz}:{views} 1 1 0 2 1 1.0 1.0 0 0 0 0 0 1\n")
    monkeypatch.setenv("LS_AUTOTUNE_CACHE", str(cache))
    f = to_dev(torch, potential(ph.random_potential_like(shape, seed=4)), torch.float32)
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    plan = ls.Plan(shape, KB, H)
    assert plan.autotune(views, f)["from_cache"] == 1
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.view_as_complex(torch.randn((views,) + shape + (2,), device="cuda", generator=g))
    y = torch.empty_like(x)
    ls.ls_profile(plan.handle, True)
    ls.ls_matvec_batch(plan.handle, f, x, y, True)
    torch.cuda.synchronize()
    times = ls.ls_profile(plan.handle, False)
    # one launch stands for the three passes: its time is divided between them 1 : 2 : 1
    assert times["fy"][0] > 0 and times["fy"][0] == times["iy"][0] == pytest.approx(times["z"][0] / 2, rel=1e-6)
    for q in (0, 1, 33, 69):
        ref = op.A(x[q].cpu().numpy().astype("complex128"), f.cpu().numpy().astype("float64"), True)
        assert rel(y[q].cpu().numpy(), ref) < 3e-6, q
    plan.close()
