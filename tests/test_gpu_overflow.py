"""Compensated sums that overflow give the infinity that a plain sum gives, not the
NaN of their carry: the FP64 boundary data (partial sums of a split contraction)
and the network's first and last weight gradients."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _skip():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    return dgx


@pytest.mark.parametrize("n,p", [(2, 4), (3, 8)])
def test_boundary_data_overflow(n, p):
    dgx = _skip()
    # on a unit cube the integral of 1 / r from a boundary point is 1.19 (corner) and
    # more: every value passes 1.6e308 * 1.19 > DBL_MAX, no term of the sums does
    s = dgx.PoissonSolver([0.0] * 3, [1.0] * 3, (n, n, n), p)
    g = s.boundary_data(torch.full((1, s.Nq), 1.6e308, device="cuda", dtype=torch.float64))
    assert bool(torch.isposinf(g).all())
    s.close()


@pytest.mark.parametrize("ne", [1, 40])
def test_weight_gradient_overflow(ne):
    dgx = _skip()
    p, n1 = 2, 3
    prm = {k: np.zeros(shape) for k, shape in dgx.NN_LAYOUT}
    prm["b1"][:] = 1.5
    prm["W2"][1, 1, 1] = 2.0 * np.eye(32)
    prm["W3"][1, 1, 1, :, 0] = 1.0
    s = dgx.PoissonSolver([-1.0] * 3, [1.0] * 3, (2, 2, 2), p, precision=dgx.DG_PREC_MIXED)
    dgx.dg_nn_set_params(s.h, dgx.nn_pack(prm))
    x = torch.ones(ne, n1 ** 3, 2, device="cuda")
    dgx.dg_nn_forward(s.h, x, save_act=True)
    g = torch.zeros_like(x)
    g[ne // 2, 13, 0] = 3e38  # the middle node: g_a1 = 2 * 3e38 and a2 * 3e38 = 9e38 overflow
    grad = dgx.nn_unpack(dgx.dg_nn_backward(s.h, x, g).cpu().numpy())
    assert np.isposinf(grad["W1"]).all()
    assert np.isposinf(grad["W3"][..., 0]).all() and not grad["W3"][..., 1].any()
    s.close()
