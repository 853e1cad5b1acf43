"""Batched calls read and write the caller's vectors in place.  Every way an output may coincide with or overlap
another vector, vectors that are only 8-byte aligned, and solves that end before their first update give the
results of separate, aligned vectors."""
import pytest

import phantoms as ph

from gpu_common import H, KB, potential, rel, to_dev, torch_and_lib

SHAPE = (16, 24, 32)
TOL = 1e-6   # the same arithmetic on the same values; a solve's sums may group differently by a few roundings


def _setup(torch, ls, views=3):
    f = to_dev(torch, potential(ph.random_ellipsoids(SHAPE, count=3, rmin=2, rmax=6, dn_max=0.04)), torch.float32)
    plan = ls.Plan(SHAPE, KB, H, tol=1e-6)
    uin = plan.plane_waves(ph.cone_directions(views, 0.8) * KB)
    return plan, f, uin


def _same(a, b):
    return rel(a.cpu().numpy(), b.cpu().numpy()) < TOL


@pytest.mark.gpu
@pytest.mark.parametrize("how", ["in place", "rotated", "one view on another", "shifted", "unaligned"])
def test_operator_outputs_over_inputs(how):
    torch, ls = torch_and_lib()
    plan, f, x = _setup(torch, ls)
    n = x[0].numel()
    ref = torch.empty_like(x)
    ls.ls_matvec_batch(plan.handle, f, x, ref)
    pool = torch.empty(4 * n + 2, dtype=torch.complex64, device="cuda")
    off = 1 if how == "unaligned" else 0
    xs = [pool[off + q * n:off + (q + 1) * n].view(SHAPE) for q in range(3)]
    for a, b in zip(xs, x):
        a.copy_(b)
    if how == "in place":
        ys = list(xs)
    elif how == "rotated":
        ys = [xs[1], xs[2], xs[0]]
    elif how == "one view on another":
        ys = [xs[0], xs[2], pool[3 * n:4 * n].view(SHAPE)]
    elif how == "shifted":
        ys = [pool[5 + q * n:5 + (q + 1) * n].view(SHAPE) for q in range(3)]
    else:
        ys = [torch.empty(n + 1, dtype=torch.complex64, device="cuda")[1:].view(SHAPE) for _ in range(3)]
    ls.ls_matvec_batch(plan.handle, f, xs, ys)
    torch.cuda.synchronize()
    for q in range(3):
        assert _same(ys[q], ref[q]), (how, q)
    plan.close()


@pytest.mark.gpu
def test_back_to_back_operator_calls_keep_their_own_vectors():
    # the calls do not synchronise: the second must not change what the first one's kernels read
    torch, ls = torch_and_lib()
    plan, f, x = _setup(torch, ls)
    refs = [torch.empty_like(x), torch.empty_like(x)]
    xs = [x, x * 2.0]
    for a, r in zip(xs, refs):
        ls.ls_matvec_batch(plan.handle, f, a, r)
        torch.cuda.synchronize()
    outs = [torch.empty_like(x) for _ in range(20)]
    for k, o in enumerate(outs):
        ls.ls_matvec_batch(plan.handle, f, xs[k % 2], o)
    torch.cuda.synchronize()
    for k, o in enumerate(outs):
        assert torch.equal(o, refs[k % 2]), k
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("how", ["in place", "next view", "unaligned", "warm in place", "warm unaligned", "far inside"])
def test_solve_outputs_over_inputs(how):
    torch, ls = torch_and_lib()
    plan, f, uin = _setup(torch, ls)
    q, n = uin.shape[0], uin[0].numel()
    u_ref, far_ref, code, _ = plan.forward(f, uin)
    assert code == ls.LS_OK
    far = plan.detector(q)
    pool = torch.empty((q + 1) * n + 2, dtype=torch.complex64, device="cuda")
    off = 1 if "unaligned" in how else 0
    us = [pool[off + k * n:off + (k + 1) * n].view(SHAPE) for k in range(q)]
    for a, b in zip(us, uin):
        a.copy_(b)
    if how == "in place":
        outs = us
    elif how == "next view":
        outs = [pool[(k + 1) * n:(k + 2) * n].view(SHAPE) for k in range(q)]
    else:
        outs = [torch.empty(n + 1, dtype=torch.complex64, device="cuda")[1 if off else 0:][:n].view(SHAPE) for _ in range(q)]
    if how == "far inside":    # the far field of view 0 lies in its field's buffer; the field wins, as written last
        far = [outs[0][0], far[1], far[2]]
    if how.startswith("warm"):
        for a, b in zip(outs, uin):
            a.copy_(b)
        code, _ = ls.ls_forward_warm(plan.handle, f, uin, outs, outs, far)
    else:
        code, _ = ls.ls_forward(plan.handle, f, us, outs, far)
    torch.cuda.synchronize()
    assert code == ls.LS_OK
    for k in range(q):
        assert _same(outs[k], u_ref[k]), (how, k)
        assert (how == "far inside" and k == 0) or _same(far[k], far_ref[k]), (how, k)
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("views", [1, 3])
def test_solve_that_starts_converged_returns_the_incident_field(views):
    torch, ls = torch_and_lib()
    plan, f, uin = _setup(torch, ls, views)
    zero = torch.zeros_like(f)
    u, far, code, stats = plan.forward(zero, uin)
    torch.cuda.synchronize()
    assert code == ls.LS_OK and all(s["iterations"] == 0 for s in stats)
    assert torch.equal(u, uin) and float(far.abs().max()) == 0.0
    # the gradient at f = 0 with recomputed forward fields: Re(conj(u_in) G~^H r)
    r = plan.detector(views)
    r.copy_(torch.randn_like(r))
    g, code, _ = plan.gradient(zero, r, u_in=uin)
    w = plan.field(views)
    ls.ls_farfield_adjoint(plan.handle, r, w)
    assert code == ls.LS_OK
    assert _same(g, (uin.conj() * w).real.sum(0))
    plan.close()
