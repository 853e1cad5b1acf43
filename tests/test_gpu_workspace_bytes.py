"""ls_workspace_bytes against the device memory that a plan holds once its workspace exists."""
import pytest

from gpu_common import H, KB, torch_and_lib

# tables and partial sums (a few hundred KB a view) and the allocator's granularity of 2 MiB for each array
SLACK = 48 << 20


@pytest.mark.gpu
@pytest.mark.parametrize("shape,views", [((128, 128, 128), 2), ((144, 144, 144), 1), ((192, 192, 128), 1),
                                         ((96, 192, 96), 2), ((64, 192, 192), 1)])
def test_estimate_is_what_a_plan_allocates(shape, views):
    torch, ls = torch_and_lib()
    nz, ny, nx = shape
    f = torch.zeros(shape, device="cuda")
    x = torch.zeros((views,) + shape, dtype=torch.complex64, device="cuda")

    def used():
        free, _ = torch.cuda.mem_get_info()
        plan = ls.Plan(shape, KB, H)
        ls.ls_matvec_batch(plan.handle, f, x, x)
        torch.cuda.synchronize()
        got = free - torch.cuda.mem_get_info()[0]
        plan.close()
        return got

    used()          # the kernels' modules are loaded once
    got = used()
    want = ls.ls_workspace_bytes((nx, ny, nz), views)
    assert abs(got - want) < SLACK, (got, want)
