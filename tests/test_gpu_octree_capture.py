"""The octree operator in CUDA graphs: a captured call owns its scratch, so two
graphs and direct calls on the same handle may overlap. Results are the same
bits as those of a call by itself."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,B", [(2, 40), (6, 70)])
def test_captured_operator_overlaps(p, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    lo, hi, n = [-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2)
    leaves = dgx.dg_octree_refine(lo, hi, n, p, lambda x: np.exp(-40.0 * np.sum((x - 0.4) ** 2, axis=1)), 1e-4, 2)
    assert len(set(leaves[:, 0].tolist())) > 1
    s = dgx.OctreeSolver(lo, hi, n, p, leaves, precond=0)
    gen = torch.Generator(device="cuda").manual_seed(5)
    us = [torch.randn(B, s.Nq, generator=gen, device="cuda", dtype=torch.float64) for _ in range(3)]
    want = [s.apply(u) for u in us]
    graphs, outs, streams = [], [], [torch.cuda.Stream() for _ in range(3)]
    for u, st in zip(us[:2], streams):
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            outs.append(s.apply(u, stream=st))
        graphs.append(g)
    torch.cuda.synchronize()
    direct = []
    for _ in range(5):
        for g, o, st in zip(graphs, outs, streams):
            with torch.cuda.stream(st):
                o.zero_()
                g.replay()
        with torch.cuda.stream(streams[2]):
            direct.append(s.apply(us[2], stream=streams[2]))
    torch.cuda.synchronize()
    for o, w in zip(outs, want):
        assert torch.equal(o, w)
    assert all(torch.equal(d, want[2]) for d in direct)
    s.close()
