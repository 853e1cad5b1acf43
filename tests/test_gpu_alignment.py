"""Vectors at an odd float offset (4-byte aligned, as ls_c64 is two floats) give the results of aligned ones in every
call that copied its vectors before it used them in place.  The pointers never reach a kernel: the library sends
such vectors through its workspace."""
import numpy as np
import pytest

import phantoms as ph

from gpu_common import H, KB, LAM, potential, rel, to_dev, torch_and_lib

SHAPE = (16, 24, 32)
VIEWS = 3
TOL = 1e-6   # the same arithmetic on the same values; a solve's sums may group differently by a few roundings


class Odd:
    """VIEWS vectors of `shape`, each at an odd float offset of one buffer, with a guard float on either side."""

    def __init__(self, torch, shape, values=None):
        self.n, self.shape = int(np.prod(shape)), tuple(shape)
        self.step = 2 * self.n + 4
        self.buf = torch.full((VIEWS * self.step + 4,), 7.0, device="cuda")
        assert self.buf.data_ptr() % 16 == 0
        if values is not None:
            for q in range(VIEWS):
                self._floats(q).copy_(torch.view_as_real(values[q]).flatten())

    def _floats(self, q):
        return self.buf[1 + q * self.step:1 + q * self.step + 2 * self.n]

    @property
    def ptrs(self):
        p = [self._floats(q).data_ptr() for q in range(VIEWS)]
        assert all(v % 8 == 4 for v in p)
        return p

    def __getitem__(self, q):
        assert float(self.buf[q * self.step]) == 7.0 and float(self.buf[1 + q * self.step + 2 * self.n]) == 7.0
        v = self._floats(q).cpu().numpy()
        return (v[0::2] + 1j * v[1::2]).reshape(self.shape)


def _setup(torch, ls):
    f = to_dev(torch, potential(ph.random_ellipsoids(SHAPE, count=3, rmin=2, rmax=6, dn_max=0.04)), torch.float32)
    plan = ls.Plan(SHAPE, KB, H, tol=1e-6)
    return plan, f, plan.plane_waves(ph.cone_directions(VIEWS, 0.8) * KB)


def _same(odd, ref):
    for q in range(VIEWS):
        assert rel(odd[q], ref[q].cpu().numpy()) < TOL, q


@pytest.mark.gpu
@pytest.mark.parametrize("odd", ["x", "y", "both", "in place"])
def test_batched_operator(odd):
    torch, ls = torch_and_lib()
    plan, f, x = _setup(torch, ls)
    ref = torch.empty_like(x)
    ls.ls_matvec_batch(plan.handle, f, x, ref)
    xo, yo, y = Odd(torch, SHAPE, x), Odd(torch, SHAPE), torch.empty_like(x)
    ls.ls_matvec_batch(plan.handle, f, list(x) if odd == "y" else xo.ptrs,
                       list(y) if odd == "x" else xo.ptrs if odd == "in place" else yo.ptrs)
    torch.cuda.synchronize()
    if odd == "x":
        assert torch.equal(y, ref)
    else:
        _same(xo if odd == "in place" else yo, ref)
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("pupil", [False, True])
@pytest.mark.parametrize("warm", [False, True])
def test_solve(warm, pupil):
    torch, ls = torch_and_lib()
    plan, f, uin = _setup(torch, ls)
    if pupil:
        ls.ls_set_pupil(plan.handle, 2 * np.pi * 0.9 / LAM, -1.7)
    u_ref, far_ref, code, _ = plan.forward(f, uin)
    assert code == ls.LS_OK
    a, u, far = Odd(torch, SHAPE, uin), Odd(torch, SHAPE, uin), Odd(torch, SHAPE[1:])
    if warm:
        code, _ = ls.ls_forward_warm(plan.handle, f, a.ptrs, u.ptrs, u.ptrs, far.ptrs)
    else:
        code, _ = ls.ls_forward(plan.handle, f, a.ptrs, u.ptrs, far.ptrs)
    torch.cuda.synchronize()
    assert code == ls.LS_OK
    _same(u, u_ref)
    _same(far, far_ref)
    # the gradient recomputes its forward fields from u_in
    r = torch.randn_like(far_ref)
    g_ref, code, _ = plan.gradient(f, r, u_in=uin)
    assert code == ls.LS_OK
    g = torch.empty_like(f)
    code, _ = ls.ls_gradient(plan.handle, f, r, g, u_in=a.ptrs)
    torch.cuda.synchronize()
    assert code == ls.LS_OK and rel(g.cpu().numpy(), g_ref.cpu().numpy()) < TOL
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("pupil", [False, True])
def test_far_field_and_adjoint(pupil):
    torch, ls = torch_and_lib()
    plan, f, u = _setup(torch, ls)
    if pupil:
        ls.ls_set_pupil(plan.handle, 2 * np.pi * 0.9 / LAM, -1.7)
    far_ref, back_ref = plan.detector(VIEWS), plan.field(VIEWS)
    ls.ls_farfield(plan.handle, f, u, far_ref)
    ls.ls_farfield_adjoint(plan.handle, far_ref, back_ref)
    far, back = Odd(torch, SHAPE[1:]), Odd(torch, SHAPE)
    ls.ls_farfield(plan.handle, f, Odd(torch, SHAPE, u).ptrs, far.ptrs)
    ls.ls_farfield_adjoint(plan.handle, far_ref, back.ptrs)
    torch.cuda.synchronize()
    _same(far, far_ref)
    _same(back, back_ref)
    plan.close()
