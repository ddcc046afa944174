"""Work split of the Schwarz smoother by count: the gather takes sources in groups of
up to four (FP32) and two (FP64). A source's result does not depend on it, bit for
bit; the values are in test_gpu_parity.py."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI = [-2.0, -1.0, 0.5], [2.0, 1.5, 2.0]


@pytest.mark.parametrize("n,p", [((3, 2, 4), 2), ((2, 3, 2), 4), ((3, 3, 3), 7)])
@pytest.mark.parametrize("fp32", [False, True])
def test_smoother_source_groups(n, p, fp32):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    dt = torch.float32 if fp32 else torch.float64
    s = dgx.PoissonSolver(LO, HI, n, p, precision=dgx.DG_PREC_MIXED if fp32 else dgx.DG_PREC_FP64)
    r = torch.randn(9, s.Nq, generator=torch.Generator(device="cuda").manual_seed(9), device="cuda", dtype=dt)
    z = s.smoother(r)
    for B in range(1, 9):
        assert torch.equal(s.smoother(r[:B].contiguous()), z[:B])
    s.close()
