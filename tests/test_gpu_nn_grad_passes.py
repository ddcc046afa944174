"""The exact weight gradients of test_gpu_nn_grad_exact.py at the degrees where a block
takes one element at a time, with more elements than blocks (a block reloads over the
last element's gradients and carries its sums on) and a last pass that is not full.
Same inputs, reference and tolerance as there."""

import pytest

pytest.importorskip("torch")
import test_gpu_nn_grad_exact as exact  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,ne", [(6, 200), (6, 700), (7, 153), (7, 700)])
def test_gradients_over_several_passes(p, ne):
    exact.test_first_and_last_layer_gradients(p, ne)
