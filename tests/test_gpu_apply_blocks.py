"""FP64 operator forms by element count: the direct blocks of p = 1 and 2, blocks of
two sizes at p = 5 and 6, and the small form, on both sides of the lines between
them, against the dense Kronecker oracle (1e-13 of the largest entry, as in
test_gpu_parity.py). A field's result does not depend on the batch."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI = [-2.0, -1.0, 0.5], [2.0, 1.5, 2.0]


@pytest.mark.parametrize("n,p,B", [((1, 1, 1), 1, 1), ((2, 1, 3), 1, 1), ((5, 4, 3), 1, 33), ((5, 4, 3), 1, 700),
                                   ((1, 1, 2), 2, 3), ((3, 4, 5), 2, 10), ((3, 4, 5), 2, 12), ((3, 4, 5), 2, 401),
                                   ((5, 3, 3), 5, 9), ((5, 3, 3), 5, 10), ((5, 3, 3), 5, 17), ((5, 3, 3), 5, 34),
                                   ((4, 4, 3), 6, 13), ((4, 4, 3), 6, 32), ((4, 4, 3), 6, 45)])
def test_fp64_operator_blocks(n, p, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    m = oracle.Mesh(LO, HI, n, p)
    s = dgx.PoissonSolver(LO, HI, n, p)
    u = torch.randn(B, m.Nq, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda", dtype=torch.float64)
    out = s.apply(u)
    A = oracle.assemble_kron(m)
    pick = sorted({0, B // 2, B - 1})
    ref = (A @ u[pick].cpu().numpy().T).T
    err = np.abs(out[pick].cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= 1e-13, err
    for k in pick:
        assert torch.equal(s.apply(u[k:k + 1].contiguous())[0], out[k])
    s.close()
