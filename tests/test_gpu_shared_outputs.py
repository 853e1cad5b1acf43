"""Far fields and adjoint far fields whose outputs overlap: the last view's stands, as when each view was copied out
in turn."""
import pytest

import phantoms as ph

from gpu_common import H, KB, potential, rel, to_dev, torch_and_lib

VIEWS = 24


@pytest.mark.gpu
@pytest.mark.parametrize("shift", [0, 1, 100])
@pytest.mark.parametrize("what", ["far", "adjoint"])
def test_last_view_stands(what, shift):
    torch, ls = torch_and_lib()
    shape = (16, 48, 48)
    plan = ls.Plan(shape, KB, H)
    f = to_dev(torch, potential(ph.random_potential_like(shape, seed=4)), torch.float32)
    g = torch.Generator(device="cuda").manual_seed(5)
    small = what == "far"
    x = torch.view_as_complex(torch.randn((VIEWS,) + (shape if small else shape[1:]) + (2,), device="cuda", generator=g))
    ref = plan.detector(VIEWS) if small else plan.field(VIEWS)

    def call(out):
        if small:
            ls.ls_farfield(plan.handle, f, x, out)
        else:
            ls.ls_farfield_adjoint(plan.handle, x, out)
        torch.cuda.synchronize()

    call(ref)
    n = ref[0].numel()
    pool, want = (torch.zeros(n + shift * VIEWS, dtype=torch.complex64, device="cuda") for _ in range(2))
    for q in range(VIEWS):
        want[shift * q:shift * q + n].copy_(ref[q].flatten())
    for _ in range(5):
        call([pool[shift * q:shift * q + n] for q in range(VIEWS)])
        assert rel(pool.cpu().numpy(), want.cpu().numpy()) < 1e-6
    plan.close()
