"""Weight gradients of layers 1 and 3 (FP32 operands as three BF16 parts on the
tensor cores) against float64 sums, with parameters for which every BF16
activation and gradient is exact: W1 = 0, b1 = 1.5 (a1 = 1.5), W2 the identity at
the centre tap, b2 = 0.5 (a2 = 2), W3 one at the centre tap of channel 0, output
gradients of channel 0 that are BF16 numbers. What is left is the FP32 summation:
chains of at most 32 MMA steps of 2^-24 each, joined to compensated sums, hence
2e-6 of the largest entry. 2000 elements are worked in groups at small degrees,
the last one not full."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("ne", [1, 60, 2000])
def test_first_and_last_layer_gradients(p, ne):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    n1 = p + 1
    prm = {k: np.zeros(shape) for k, shape in dgx.NN_LAYOUT}
    prm["b1"][:] = 1.5
    prm["W2"][1, 1, 1] = np.eye(32)
    prm["b2"][:] = 0.5
    prm["W3"][1, 1, 1, :, 0] = 1.0
    s = dgx.PoissonSolver([-1.0] * 3, [1.0] * 3, (2, 2, 2), p, precision=dgx.DG_PREC_MIXED)
    dgx.dg_nn_set_params(s.h, dgx.nn_pack(prm))
    rng = np.random.default_rng(p)
    x = rng.standard_normal((ne, n1 ** 3, 2)).astype(np.float32)
    g = rng.standard_normal((ne, n1 ** 3, 2)).astype(np.float32)
    g[..., 0] = torch.tensor(g[..., 0]).bfloat16().float().numpy()
    xd, gd = torch.tensor(x, device="cuda"), torch.tensor(g, device="cuda")
    out = dgx.dg_nn_forward(s.h, xd, save_act=True).cpu().numpy()
    assert np.abs(out[..., 0] - 64.0).max() <= 1e-4 and not out[..., 1].any()
    grad = dgx.nn_unpack(dgx.dg_nn_backward(s.h, xd, gd).cpu().numpy())
    pad = np.zeros((ne, n1 + 2, n1 + 2, n1 + 2, 2))
    inner = pad[:, 1:-1, 1:-1, 1:-1]
    x5, g5 = (v.astype(np.float64).reshape(ne, n1, n1, n1, 2) for v in (x, g))
    dW1, dW3 = np.zeros((3, 3, 3, 2, 32)), np.zeros((3, 3, 3, 32, 2))
    for v, dW, sign in ((x5, dW1, 1), (g5, dW3, -1)):
        inner[:] = v
        for t in np.ndindex(3, 3, 3):
            o = [1 + sign * (k - 1) for k in t]
            sh = pad[:, o[0]:o[0] + n1, o[1]:o[1] + n1, o[2]:o[2] + n1]
            if sign > 0:  # in[n + t] g_a1[n], g_a1 = g of channel 0 for every channel
                dW[t] = np.einsum("ezyxi,ezyx->i", sh, g5[..., 0])[:, None]
            else:  # g3[n - t] a2[n], a2 = 2
                dW[t] = 2.0 * sh.sum(axis=(0, 1, 2, 3))[None, :]
    for name, ref in (("W1", dW1), ("W3", dW3)):
        err = np.abs(grad[name] - ref).max() / np.abs(ref).max()
        assert err <= 2e-6, (name, err)
    s.close()
