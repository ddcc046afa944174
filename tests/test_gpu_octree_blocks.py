"""Leaf-block inverse of the octree at every degree, with few fields (one leaf per
block) and many: P r is checked leaf by leaf against the diagonal blocks that the
operator itself gives on unit fields (the operator is checked against the dense
oracle in test_gpu_octree.py). Tolerance 1e-11 of the right-hand side's largest
entry, as for the leaf blocks in test_gpu_octree_solve.py; a field's result does
not depend on the batch."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("form", [0, 1])
def test_leaf_block_inverse(p, form):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()

    def rho(x):
        return np.exp(-40.0 * np.sum((x - np.array([-0.6, -0.5, 0.4])) ** 2, axis=1))

    lo, hi, n = [-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (2, 1, 1)
    leaves = dgx.dg_octree_refine(lo, hi, n, p, rho, 1e-5, 1)
    E, npe = leaves.shape[0], (p + 1) ** 3
    s = dgx.OctreeSolver(lo, hi, n, p, leaves, penalty_form=form, precond=0)
    B = 1 + 2 * 152 * 64 // E
    g = torch.Generator(device="cuda").manual_seed(6)
    r = torch.randn(B, s.Nq, generator=g, device="cuda", dtype=torch.float64)
    z = s.precond(r)
    for k in (0, B - 1):
        assert torch.equal(s.precond(r[k:k + 1].contiguous())[0], z[k])
    for e in sorted({0, E // 2, E - 1}):
        u = torch.zeros(npe, s.Nq, device="cuda", dtype=torch.float64)
        u[:, e * npe:(e + 1) * npe] = torch.eye(npe, device="cuda", dtype=torch.float64)
        block = s.apply(u)[:, e * npe:(e + 1) * npe]  # row j: column j of A's diagonal block
        back = z[0, e * npe:(e + 1) * npe] @ block
        want = r[0, e * npe:(e + 1) * npe]
        assert float((back - want).abs().max()) <= 1e-11 * float(want.abs().max()), e
    s.close()
