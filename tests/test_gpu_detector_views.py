"""Detector-plane operators for several views in one call against the FP64 oracle: the far field and its adjoint where
slices are summed in several chunks and in one, and the pupil P and P^H (in place and out of place) on detectors
whose padded lengths take one to eight pencils per CTA, with row counts that do not fill a CTA."""
import numpy as np
import pytest

import phantoms as ph
from oracle import incident, model

from gpu_common import ETA_B, H, KB, LAM, potential, rel, to_dev, torch_and_lib

# float32 storage and sums of at most 192 slices of 2-D transforms (2 log2 of the padded plane <= 34 additions):
# 6e-8 * (192 ** 0.5 + 34) < 3e-6
TOL = 3e-6
# float64 transforms, one rounding to float32 at the end
TOL_PUPIL = 2e-7


@pytest.mark.gpu
@pytest.mark.parametrize("shape,views", [((8, 8, 8), 1), ((48, 24, 16), 1), ((16, 24, 32), 5), ((192, 16, 24), 2),
                                         ((12, 72, 48), 3)])
def test_far_field_and_adjoint(shape, views):
    torch, ls = torch_and_lib()
    f64 = potential(ph.random_potential_like(shape, seed=5))
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    plan = ls.Plan(shape, KB, H)
    f = to_dev(torch, f64, torch.float32)
    f64 = f.cpu().numpy().astype(np.float64)
    u = torch.stack([to_dev(torch, ph.random_field(shape, q), torch.complex64) for q in range(views)])
    r = torch.stack([to_dev(torch, ph.random_field(shape[1:], 50 + q), torch.complex64) for q in range(views)])
    far, back = plan.detector(views), plan.field(views)
    ls.ls_farfield(plan.handle, f, u, far)
    ls.ls_farfield_adjoint(plan.handle, r, back)
    for q in range(views):
        assert rel(far[q].cpu().numpy(), op.farfield_fft(f64 * u[q].cpu().numpy().astype(np.complex128))) < TOL
        assert rel(back[q].cpu().numpy(), op.farfield_adjoint_fft(r[q].cpu().numpy().astype(np.complex128))) < TOL
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("ny,nx", [(8, 8), (12, 48), (72, 24), (144, 128), (192, 16)])
@pytest.mark.parametrize("in_place", [False, True])
def test_pupil_on_several_views(ny, nx, in_place):
    torch, ls = torch_and_lib()
    views, kcut, dist = 3, 2 * np.pi * 0.9 / LAM, -1.7
    plan = ls.Plan((8, ny, nx), KB, H)
    ls.ls_set_pupil(plan.handle, kcut, dist)
    y = torch.stack([to_dev(torch, ph.random_field((ny, nx), q), torch.complex64) for q in range(views)])
    y64 = y.cpu().numpy().astype(np.complex128)
    Hd = incident.pupil_transfer((ny, nx), H, KB, kcut, dist)
    for adjoint in (False, True):
        src = y.clone()
        out = src if in_place else torch.empty_like(src)
        ls.ls_apply_pupil(plan.handle, src, out, adjoint)
        torch.cuda.synchronize()
        for q in range(views):
            ref = incident.apply_pupil(y64[q], Hd, adjoint=adjoint)
            assert rel(out[q].cpu().numpy(), ref) < TOL_PUPIL, (q, adjoint)
    plan.close()
