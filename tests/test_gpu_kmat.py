"""The K contraction at the edges of its two kernels (all N^2 outputs in one block
up to 16 orbitals, 32 x 32 tiles beyond): K_ij = sum_q W_q psi_i (W psi_j) with
W psi_j = -X psi_j from the J/K action on the orbitals themselves, which does not
use the contraction. 1e-9 relative to the largest entry (both sides solve to
rtol 1e-12; the fixed-order sums agree to round-off)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 11, 15, 16, 17, 33])
@pytest.mark.parametrize("n,p", [((2, 1, 1), 2), ((4, 4, 4), 4)])
def test_kmat_edges(N, n, p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    s = dgx.PoissonSolver([-3.0] * 3, [3.0] * 3, n, p, rtol=1e-12)
    xyz, w = s.node_coords()
    rng = np.random.default_rng(N)
    c = rng.uniform(-1.0, 1.0, size=(N, 3))
    psi = np.stack([np.exp(-np.sum((xyz - ci) ** 2, axis=1)) * (1.0 + 0.1 * k) for k, ci in enumerate(c)])
    d = torch.tensor(psi, device="cuda")
    K, eh, ex, st = s.exchange_build(d)
    _, XU, _ = s.jk_apply(d, d, hartree=False)
    ref = -(psi * w) @ XU.cpu().numpy().T
    assert np.abs(K - ref).max() <= 1e-9 * np.abs(ref).max()
    s.close()
