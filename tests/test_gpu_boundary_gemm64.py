"""FP64 Gaussian-sum boundary data at the edges of its GEMM tiles: 2 to 65
nodes an axis (one short tile, exactly one, one row or column more), with and
without a split contraction, against the direct quadrature. Tolerance as in
test_gpu_parity.py::test_boundary_data: 3e-12 of sum |W f| / r (the Gaussian
sum's 1e-12 and the round-off of three contractions)."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [((1, 16, 15), 1), ((11, 1, 10), 2), ((13, 1, 6), 4), ((1, 1, 1), 1), ((4, 2, 3), 7)])
@pytest.mark.parametrize("B", [1, 5])
def test_boundary_data_tile_edges(n, p, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    lo, hi = [-4.0, -3.0, -3.5], [4.0, 3.5, 3.0]
    m = oracle.Mesh(lo, hi, n, p)
    f = np.random.default_rng(11).standard_normal((B, m.Nq))
    s = dgx.PoissonSolver(lo, hi, n, p)
    g = s.boundary_data(torch.tensor(f, device="cuda"), route=1).cpu().numpy()
    ref = np.concatenate([a.transpose(0, 2, 1).reshape(B, -1) for a in oracle.boundary_data_direct(m, f)], axis=1)
    bound = np.concatenate([a.transpose(0, 2, 1).reshape(B, -1) for a in oracle.boundary_data_direct(m, np.abs(f))],
                           axis=1)
    assert g.shape == ref.shape
    assert (np.abs(g - ref) <= 3e-12 * bound.max()).all()
    s.close()
