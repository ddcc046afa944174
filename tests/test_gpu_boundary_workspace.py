"""The boundary data's split-K partials: as large as the mesh and the batch need (one
source of a 4^3, p = 4 mesh: under 1 MB) and part of the workspace that the handle
reports. Device allocations come in blocks of 2 MB."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.mark.parametrize("n,p,B,most", [(4, 4, 1, 16), (1, 1, 3, 16), (8, 6, 2, 64)])
def test_boundary_workspace(n, p, B, most):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    s = dgx.PoissonSolver([-4.0] * 3, [4.0] * 3, (n, n, n), p)
    f = torch.rand(B, s.Nq, device="cuda", dtype=torch.float64)
    s.boundary_data(f[:1], dgx.DG_BC_DIRECT)  # modules and common workspace
    torch.cuda.synchronize()
    free0, ws0 = torch.cuda.mem_get_info()[0], dgx.dg_get_info(s.h).workspace_bytes
    s.boundary_data(f)
    torch.cuda.synchronize()
    taken, told = free0 - torch.cuda.mem_get_info()[0], dgx.dg_get_info(s.h).workspace_bytes - ws0
    assert taken <= most * MB
    assert told >= 0 and taken - told <= 16 * MB  # eight buffers, each rounded up to 2 MB
    s.close()
