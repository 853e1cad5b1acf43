"""A solve whose views have all converged at its start: on large batches only the residual is evaluated; with a small
one a chunk of iterations goes out with it, in which the views are masked off.  Read from the NVTX ranges."""
import pytest

from gpu_common import torch_and_lib
from test_trace import _run

CODE = """
    import torch
    import paper_1910_13844_gb300 as ls
    shape, views = {shape}, {views}
    plan = ls.Plan(shape, 8.0, 0.1, use_graphs=0)
    f = torch.zeros(shape, device="cuda")
    u = torch.ones((views,) + shape, dtype=torch.complex64, device="cuda")
    out = torch.empty_like(u)
    code, stats = ls.ls_forward(plan.handle, f, u, out)
    torch.cuda.synchronize()
    assert code == ls.LS_OK and all(s["iterations"] == 0 and s["matvecs"] == 1 for s in stats), stats
    assert torch.equal(u, out)
    plan.close()
"""


@pytest.mark.gpu
@pytest.mark.parametrize("shape,views,most", [((192, 192, 128), 1, 1), ((64, 64, 64), 16, 1), ((64, 64, 64), 15, 5),
                                              ((16, 16, 16), 2, 5)])
def test_operator_applications(tmp_path, shape, views, most):
    torch_and_lib()
    lines = _run(tmp_path, CODE.format(shape=shape, views=views))
    assert lines[lines.index("push solve"):].count("push FX") == most
