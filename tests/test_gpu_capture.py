"""Calls that do not synchronise, captured by the caller into a CUDA graph: a replay does what the call did, on what
the vectors hold by then, whatever else the plan and the host's memory were used for in between."""
import numpy as np
import pytest

import phantoms as ph

from gpu_common import H, KB, LAM, potential, to_dev, torch_and_lib

SHAPE = (16, 24, 32)


def _capture(torch, call):
    call()   # the workspace and the tables exist before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        call()
    return graph


def _use_host_memory():
    # blocks of the sizes a call's own arrays have, filled with something else
    return [np.full(n, 0x5A, dtype=np.uint8) for n in (64, 256, 512, 1024, 1 << 16) for _ in range(200)]


@pytest.mark.gpu
@pytest.mark.parametrize("views", [3, 130])
@pytest.mark.parametrize("how", ["apart", "rotated"])
def test_replayed_batched_operator(views, how):
    torch, ls = torch_and_lib()
    f = to_dev(torch, potential(ph.random_ellipsoids(SHAPE, count=3, rmin=2, rmax=6, dn_max=0.04)), torch.float32)
    plan = ls.Plan(SHAPE, KB, H)
    g = torch.Generator(device="cuda").manual_seed(1)
    a, b = (torch.view_as_complex(torch.randn((views,) + SHAPE + (2,), device="cuda", generator=g)) for _ in range(2))
    want = torch.empty_like(a)
    ls.ls_matvec_batch(plan.handle, f, b, want, True)
    x = list(a.clone().unbind(0))
    y = list(torch.empty_like(a).unbind(0)) if how == "apart" else x[1:] + x[:1]
    graph = _capture(torch, lambda: ls.ls_matvec_batch(plan.handle, f, x, y, True))
    ls.ls_matvec_batch(plan.handle, torch.zeros_like(f), a, torch.empty_like(a))
    keep = _use_host_memory()
    for q in range(views):
        x[q].copy_(b[q])
    graph.replay()
    torch.cuda.synchronize()
    for q in range(views):
        assert torch.equal(y[q], want[q]), q
    del keep
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("views", [3, 70])
def test_replayed_pupil(views):
    torch, ls = torch_and_lib()
    plan = ls.Plan((8, 24, 24), KB, H)
    ls.ls_set_pupil(plan.handle, 2 * np.pi * 0.9 / LAM, -1.7)
    g = torch.Generator(device="cuda").manual_seed(2)
    a, b = (torch.view_as_complex(torch.randn((views, 24, 24, 2), device="cuda", generator=g)) for _ in range(2))
    want = torch.empty_like(a)
    ls.ls_apply_pupil(plan.handle, b, want)
    x, y = a.clone(), torch.empty_like(a)
    graph = _capture(torch, lambda: ls.ls_apply_pupil(plan.handle, x, y))
    ls.ls_apply_pupil(plan.handle, a, torch.empty_like(a), True)
    keep = _use_host_memory()
    x.copy_(b)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    del keep
    plan.close()
