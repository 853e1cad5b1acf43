"""The fused y/z pass against the FP64 oracle: every y length and every z length, the pairs at the edges of its
tiles (largest tiles, rows and columns that do not fill a warp, several rounds per warp), both operators, more
views than one wave of CTAs, and pairs without a fused form, which keep the five passes."""
import pytest

import phantoms as ph
from oracle import model

from gpu_common import ETA_B, H, LAM, KB, potential, rel, to_dev, torch_and_lib

# float32 rounding of a 2-D transform pair: unit roundoff 6e-8 times about 2 log2(8 N) <= 50 additions in a chain
TOL = 3e-6

SQUARE = [(n, n) for n in (8, 12, 16, 24, 32, 48, 64, 72, 96, 128, 144)]
PAIRS = SQUARE + [(8, 192), (192, 8), (12, 144), (144, 64), (96, 192), (192, 96), (128, 72), (48, 16), (64, 24),
                  (192, 128)]


@pytest.mark.gpu
@pytest.mark.parametrize("ny,nz", PAIRS)
def test_operator_matches_the_oracle(ny, nz):
    torch, ls = torch_and_lib()
    shape = (nz, ny, 16)
    f64 = potential(ph.random_potential_like(shape, seed=ny * 1000 + nz))
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    plan = ls.Plan(shape, KB, H)
    f = to_dev(torch, f64, torch.float32)
    f64 = f.cpu().numpy().astype("float64")
    views = 3
    xs = [ph.random_field(shape, 7 * q + 1) for q in range(views)]
    x = torch.stack([to_dev(torch, v, torch.complex64) for v in xs])
    y = torch.empty_like(x)
    for adjoint in (False, True):
        ls.ls_matvec_batch(plan.handle, f, x, y, adjoint)
        torch.cuda.synchronize()
        for q in range(views):
            ref = op.A(x[q].cpu().numpy().astype("complex128"), f64, adjoint)
            assert rel(y[q].cpu().numpy(), ref) < TOL, (q, adjoint)
    one = torch.empty_like(x[0])
    ls.ls_matvec(plan.handle, f, x[2], one, True)
    torch.cuda.synchronize()
    assert rel(one.cpu().numpy(), y[2].cpu().numpy()) < TOL
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(24, 24, 24), (72, 72, 16), (64, 144, 8), (96, 72, 8)])
def test_many_views_take_several_planes_per_cta(shape):
    torch, ls = torch_and_lib()
    views = 70
    plan = ls.Plan(shape, KB, H)
    f = to_dev(torch, potential(ph.random_potential_like(shape, seed=4)), torch.float32)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.view_as_complex(torch.randn((views,) + shape + (2,), device="cuda", generator=g))
    y, one = torch.empty_like(x), torch.empty_like(x[0])
    ls.ls_matvec_batch(plan.handle, f, x, y)
    for q in (0, 1, 33, 69):
        ls.ls_matvec(plan.handle, f, x[q], one)
        torch.cuda.synchronize()
        assert rel(one.cpu().numpy(), y[q].cpu().numpy()) < TOL, q
    plan.close()
