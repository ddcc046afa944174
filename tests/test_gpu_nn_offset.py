"""Fields of the network calls at any float address: inputs, output gradients and
outputs that start 4 bytes off an 8-byte boundary give the bits of aligned ones."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _offset(t):
    """The same values, contiguous, 4 bytes off an 8-byte boundary."""
    v = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:].view(t.shape)
    assert v.data_ptr() % 8 == 4 and v.is_contiguous()
    return v.copy_(t)


@pytest.mark.parametrize("p,ne", [(1, 1), (1, 300), (4, 7), (7, 200)])
def test_network_fields_off_alignment(p, ne):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    s = dgx.PoissonSolver([-1.0] * 3, [1.0] * 3, (2, 2, 2), p, precision=dgx.DG_PREC_MIXED)
    rng = np.random.default_rng(p)
    dgx.dg_nn_set_params(s.h, (0.1 * rng.standard_normal(dgx.DG_NN_NPARAM)).astype(np.float32))
    x = torch.tensor(rng.standard_normal((ne, (p + 1) ** 3, 2)).astype(np.float32), device="cuda")
    g = torch.tensor(rng.standard_normal(x.shape).astype(np.float32), device="cuda")
    out = dgx.dg_nn_forward(s.h, x, save_act=True)
    grad = dgx.dg_nn_backward(s.h, x, g)
    for xs, gs in ((x, _offset(g)), (_offset(x), g), (_offset(x), _offset(g))):
        assert torch.equal(dgx.dg_nn_backward(s.h, xs, gs), grad)
    off = _offset(torch.zeros_like(out))
    dgx._check(dgx.load().dg_nn_forward(s.h, dgx._dev_ptr(_offset(x)), dgx._dev_ptr(off), ne, 0,
                                        dgx._stream_ptr(None)), "dg_nn_forward", s.h)
    assert torch.equal(off, out)
    s.close()
