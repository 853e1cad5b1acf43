"""The first pass at 64 points along x (eight threads a row, two transforms each in its second stage): the
transposed form of the fused pass, the plain form, and the forms that update the Krylov vectors, against the oracle."""
import pytest

import phantoms as ph
from oracle import model

from gpu_common import ETA_B, H, LAM, KB, potential, rel, to_dev, torch_and_lib

# float32 rounding of a 3-D transform pair: unit roundoff 6e-8 times about 2 log2(8 N) <= 50 additions in a chain
TOL = 3e-6


# row counts of one block, of an odd number of blocks and of many, and more views than one
@pytest.mark.gpu
@pytest.mark.parametrize("ny,nz", [(8, 8), (12, 12), (72, 8), (64, 48)])
def test_operator_and_solve_match_the_oracle(ny, nz):
    torch, ls = torch_and_lib()
    shape = (nz, ny, 64)
    plan = ls.Plan(shape, KB, H, tol=1e-6)
    f = to_dev(torch, potential(ph.random_potential_like(shape, seed=ny + nz)), torch.float32)
    f64 = f.cpu().numpy().astype("float64")
    op = model.Operator(model.setup_from_optics(shape, LAM, ETA_B, H))
    x = torch.stack([to_dev(torch, ph.random_field(shape, 7 * q + 1), torch.complex64) for q in range(3)])
    y, one = torch.empty_like(x), torch.empty_like(x[0])
    for adjoint in (False, True):
        ls.ls_matvec_batch(plan.handle, f, x, y, adjoint)
        ls.ls_matvec_noalloc(plan.handle, f, x[1], one, adjoint)
        torch.cuda.synchronize()
        for q in range(3):
            ref = op.A(x[q].cpu().numpy().astype("complex128"), f64, adjoint)
            assert rel(y[q].cpu().numpy(), ref) < TOL, (q, adjoint)
            if q == 1:
                assert rel(one.cpu().numpy(), ref) < TOL, adjoint
    # a converged solve satisfies the equation to its tolerance and the operator's rounding
    u, _, status, _ = plan.forward(f, x)
    torch.cuda.synchronize()
    assert status == 0
    for q in range(3):
        assert rel(op.A(u[q].cpu().numpy().astype("complex128"), f64, False), x[q].cpu().numpy()) < 2e-6 + TOL, q
    plan.close()
