"""Work split of the octree operator: hanging faces are taken once for both sides
by their own kernel, sources go through in chunks that its scratch holds, several
leaves share a block where there are many. The dense parity is in
test_gpu_octree.py; here a field's result does not depend on the batch (bit for
bit), a batch larger than a chunk included, nor on the streams that overlapping
calls use; and the sum over a symmetric pair <v, A u> = <u, A v> holds across
hanging faces to round-off (1e-12 of |u|_1 max |A v|)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _leaves(dgx, p, levels):
    def rho(x):
        return np.exp(-40.0 * np.sum((x - np.array([-0.6, -0.5, 0.4])) ** 2, axis=1))

    return dgx.dg_octree_refine([-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2), p, rho, 1e-4, levels)


@pytest.mark.parametrize("p,B", [(1, 700), (2, 300), (4, 40), (6, 9), (8, 600)])
@pytest.mark.parametrize("form", [0, 1])
def test_octree_operator_batches(p, B, form):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    leaves = _leaves(dgx, p, 1 if p == 8 else 2)
    assert len(set(leaves[:, 0].tolist())) > 1
    s = dgx.OctreeSolver([-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2), p, leaves, penalty_form=form, precond=0)
    g = torch.Generator(device="cuda").manual_seed(2)
    u = torch.randn(B, s.Nq, generator=g, device="cuda", dtype=torch.float64)
    out = s.apply(u)
    same = dgx.dg_octree_apply([-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2), p, leaves, u, penalty_form=form)
    assert torch.equal(out, same)
    for k in (0, B // 2, B - 1):
        assert torch.equal(s.apply(u[k:k + 1].contiguous())[0], out[k])
    a, b = float(u[0] @ out[1]), float(u[1] @ out[0])
    assert abs(a - b) <= 1e-12 * float(u[0].abs().sum() * out[1].abs().max())
    # calls that overlap on two streams
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    res = []
    for i in range(6):
        with torch.cuda.stream(streams[i % 2]):
            res.append(s.apply(u, stream=streams[i % 2]))
    torch.cuda.synchronize()
    assert all(torch.equal(r, out) for r in res)
    s.close()
