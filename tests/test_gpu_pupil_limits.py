"""ls_apply_pupil where it cannot take all views at once: no memory for their scratch, or views that share memory."""
import numpy as np
import pytest

import phantoms as ph

from gpu_common import H, KB, LAM, to_dev, torch_and_lib


def _plan(torch, ls, views, m=24):
    plan = ls.Plan((8, m, m), KB, H)
    ls.ls_set_pupil(plan.handle, 2 * np.pi * 0.9 / LAM, -1.7)
    y = torch.stack([to_dev(torch, ph.random_field((m, m), q), torch.complex64) for q in range(views)])
    return plan, y


@pytest.mark.gpu
@pytest.mark.parametrize("views,failures", [(5, 1), (5, 3), (70, 6)])
def test_scratch_for_fewer_views(views, failures):
    torch, ls = torch_and_lib()
    plan, y = _plan(torch, ls, views)
    want, got = torch.empty_like(y), torch.empty_like(y)
    ls.ls_apply_pupil(plan.handle, y, want)
    ls.ls_debug_inject(None, ls.LS_INJECT_ALLOC_FAIL, failures)
    ls.ls_apply_pupil(plan.handle, y, got)
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    # every failure was met there: the workspace of a new plan is allocated
    other = ls.Plan((8, 8, 8), KB, H)
    other.plane_waves(np.array([[0.0, 0.0, KB]]))
    other.close()
    plan.close()


@pytest.mark.gpu
def test_no_scratch_at_all():
    torch, ls = torch_and_lib()
    plan, y = _plan(torch, ls, 2)
    ls.ls_debug_inject(None, ls.LS_INJECT_ALLOC_FAIL, 2)
    with pytest.raises(ls.LsError) as err:
        ls.ls_apply_pupil(plan.handle, y, torch.empty_like(y))
    assert err.value.code == ls.LS_ENOMEM
    ls.ls_apply_pupil(plan.handle, y, y)
    torch.cuda.synchronize()
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("how", ["chain", "one output", "shifted", "both in place"])
def test_views_that_share_memory_run_in_order(how):
    torch, ls = torch_and_lib()
    m = 24

    def vectors():
        pool = torch.view_as_complex(torch.randn((5 * m * m, 2), device="cuda", generator=torch.Generator("cuda").manual_seed(3)))
        v = [pool[q * m * m:(q + 1) * m * m] for q in range(5)]
        if how == "chain":
            return pool, v[:4], v[1:]
        if how == "one output":
            return pool, v[:3], [v[4]] * 3
        if how == "shifted":
            return pool, v[1:4], [pool[q * m * m + m:(q + 1) * m * m + m] for q in range(3)]
        return pool, [v[0], v[0]], [v[0], v[0]]

    plan, _ = _plan(torch, ls, 1)
    want, x, y = vectors()
    for a, b in zip(x, y):
        ls.ls_apply_pupil(plan.handle, [a], [b])
    got, x, y = vectors()
    ls.ls_apply_pupil(plan.handle, x, y)
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    plan.close()
