"""FP32 boundary-data GEMM with few rows: at most 8, at most 16 and more rows run
on different kernels that round alike. On an octree (a row per source) a source's
mixed solve gives the same bits in batches of 1 to 17 sources; on uniform meshes
with 2 to 16 nodes an axis (a row per node) the boundary data stay within 1e-5 of
sum |W f| / r, as in test_gpu_parity.py::test_boundary_data_fp32_route_bound."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    return dgx


def test_octree_sources_by_batch(dgx):
    lo, hi, n, p = [-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2), 3

    def rho(x):
        return np.exp(-40.0 * np.sum((x - np.array([-0.6, -0.5, 0.4])) ** 2, axis=1))

    leaves = dgx.dg_octree_refine(lo, hi, n, p, rho, 1e-4, 2)
    s = dgx.OctreeSolver(lo, hi, n, p, leaves, rtol=1e-10, precision=dgx.DG_PREC_MIXED)
    g = torch.Generator(device="cuda").manual_seed(4)
    f = torch.randn(17, s.Nq, generator=g, device="cuda", dtype=torch.float64)
    v, _ = s.solve(f)
    for B in (1, 2, 8, 9, 16):
        w, _ = s.solve(f[:B].contiguous())
        assert torch.equal(w, v[:B]), B
    s.close()


@pytest.mark.parametrize("n,p", [((1, 1, 1), 1), ((1, 1, 1), 8), ((4, 2, 3), 3), ((2, 5, 8), 1)])
def test_uniform_boundary_data_few_nodes(dgx, n, p):
    lo, hi = [-4.0, -3.0, -3.5], [4.0, 3.5, 3.0]
    m = oracle.Mesh(lo, hi, n, p)
    f = np.random.default_rng(12).standard_normal((3, m.Nq))
    s = dgx.PoissonSolver(lo, hi, n, p, precision=dgx.DG_PREC_MIXED)
    g = s.boundary_data(torch.tensor(f, device="cuda"), route=1).cpu().numpy()
    ref = np.concatenate([a.transpose(0, 2, 1).reshape(3, -1) for a in oracle.boundary_data_direct(m, f)], axis=1)
    bound = np.concatenate([a.transpose(0, 2, 1).reshape(3, -1) for a in oracle.boundary_data_direct(m, np.abs(f))],
                           axis=1)
    assert (np.abs(g - ref) <= 1e-5 * bound.max()).all()
    s.close()
