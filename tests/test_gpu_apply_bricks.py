"""The operator's work split against the dense Kronecker oracle: bricks of
2 x 2 x 2 elements (chosen in FP32 when enough of them fill the chip) and single
elements, with odd element counts (bricks that lack elements), one element an
axis (both faces on the boundary), every degree, and fields that do not start on
a 16-byte boundary. Tolerances as in test_gpu_parity.py: 1e-13 (FP64) and 2e-5
(FP32) of the result's largest entry."""

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# B such that nact * bricks reaches the line of the brick rule in the first rows, and not in the last
@pytest.mark.parametrize("n,p,B", [((4, 6, 4), 1, 3000), ((5, 7, 3), 2, 600), ((3, 4, 5), 3, 300), ((5, 3, 4), 4, 120),
                                   ((5, 4, 5), 5, 30), ((4, 5, 3), 6, 40), ((7, 5, 3), 7, 24), ((5, 5, 4), 8, 24),
                                   ((1, 2, 3), 4, 3), ((1, 1, 1), 6, 2), ((3, 3, 3), 7, 2)])
@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("offset", [0, 1])
def test_operator_bricks(n, p, B, fp32, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    lo, hi = [-2.0, -1.0, 0.5], [2.0, 1.5, 2.0]
    m = oracle.Mesh(lo, hi, n, p)
    dt = torch.float32 if fp32 else torch.float64
    s = dgx.PoissonSolver(lo, hi, n, p, precision=dgx.DG_PREC_MIXED if fp32 else dgx.DG_PREC_FP64)
    g = torch.Generator(device="cuda").manual_seed(5)
    flat = torch.randn(B * m.Nq + offset, generator=g, device="cuda", dtype=dt)
    u = flat[offset:].reshape(B, m.Nq)
    out = s.apply(u).double().cpu().numpy()
    A = oracle.assemble_kron(m)
    pick = sorted({0, B // 2, B - 1})
    ref = (A @ u[pick].double().cpu().numpy().T).T
    err = np.abs(out[pick] - ref).max() / np.abs(ref).max()
    assert err <= (2e-5 if fp32 else 1e-13), err
    # the work split changes with the number of fields, the result of a field does not
    for k in pick:
        assert torch.equal(s.apply(u[k:k + 1].contiguous())[0], torch.from_numpy(out[k]).to("cuda", dt))
    s.close()
