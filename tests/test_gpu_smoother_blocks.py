"""Work split of the Schwarz smoother by count: the gather takes sources in groups of
up to four (FP32) and two (FP64), and FP64 patch solves at p = 6 and 7 change between
one patch per block (two lanes per line, or one) and several. A source's result does
not depend on it, bit for bit; the values are in test_gpu_patch_classes.py and
test_gpu_parity.py."""

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


@pytest.mark.parametrize("n,p,Bs", [((3, 4, 5), 6, (1, 9, 12, 26)), ((3, 3, 3), 7, (1, 19, 20, 33, 50, 140))])
def test_fp64_patch_blocks(n, p, Bs):
    """Patch solves by count: one patch per block with two lanes per line, one with one, several."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    s = dgx.PoissonSolver(LO, HI, n, p)
    r = torch.randn(max(Bs), s.Nq, generator=torch.Generator(device="cuda").manual_seed(11), device="cuda",
                    dtype=torch.float64)
    zp = s.patch_solves(r)
    for B in Bs:
        assert torch.equal(s.patch_solves(r[:B].contiguous()), zp[:B])
    s.close()
