"""dg_octree_operator beside other work. A captured call is one kernel node without
scratch: its graph can be instantiated more than once, with replays that overlap,
and can be a child of another graph; its results are the bits of the direct call at
every degree. A direct call does not wait for one on another stream."""

import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LO, HI, N = [-2.0, -1.0, -1.0], [2.0, 1.5, 1.0], (3, 2, 2)


def _leaves(dgx, p):
    def rho(x):
        return np.exp(-40.0 * np.sum((x - 0.4) ** 2, axis=1))

    leaves = dgx.dg_octree_refine(LO, HI, N, p, rho, 1e-4 if p < 4 else 1e-7, 2 if p < 7 else 1)
    assert len(set(leaves[:, 0].tolist())) > 1
    return leaves


class _Driver:
    """The CUDA driver's calls; every one has to succeed."""

    lib = C.CDLL("libcuda.so.1") if torch.cuda.is_available() else None

    def __getattr__(self, name):
        def call(*args):
            code = getattr(self.lib, name)(*args)
            assert code == 0, (name, code)

        return call


def _capture(cu, s, u, out, stream):
    """The graph of one captured call."""
    graph, h = C.c_void_p(), C.c_void_p(stream.cuda_stream)
    cu.cuStreamBeginCapture_v2(h, 1)
    try:
        s.apply(u, out, stream=stream)
    finally:
        cu.cuStreamEndCapture(h, C.byref(graph))
    return graph


def _setup(p, form=0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    s = dgx.OctreeSolver(LO, HI, N, p, _leaves(dgx, p), penalty_form=form, precond=0)
    u = torch.randn(5, s.Nq, generator=torch.Generator(device="cuda").manual_seed(p), device="cuda", dtype=torch.float64)
    return s, u, s.apply(u)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
def test_captured_call(p, form):
    s, u, want = _setup(p, form)
    out = torch.zeros_like(u)
    torch.cuda.synchronize()
    cu, st = _Driver(), torch.cuda.Stream()
    graph, ex, n = _capture(cu, s, u, out, st), C.c_void_p(), C.c_size_t()
    cu.cuGraphGetNodes(graph, None, C.byref(n))
    cu.cuGraphInstantiateWithFlags(C.byref(ex), graph, C.c_ulonglong(0))
    cu.cuGraphLaunch(ex, C.c_void_p(st.cuda_stream))
    torch.cuda.synchronize()
    cu.cuGraphExecDestroy(ex)
    cu.cuGraphDestroy(graph)
    assert n.value == 1
    assert torch.equal(out, want)
    s.close()


def test_captured_call_in_other_graphs():
    s, u, want = _setup(4)
    out = torch.zeros_like(u)
    torch.cuda.synchronize()
    cu = _Driver()
    st = [torch.cuda.Stream() for _ in range(2)]
    h = [C.c_void_p(x.cuda_stream) for x in st]
    graph, parent, node = _capture(cu, s, u, out, st[0]), C.c_void_p(), C.c_void_p()
    execs = [C.c_void_p() for _ in range(3)]
    cu.cuGraphCreate(C.byref(parent), 0)
    cu.cuGraphAddChildGraphNode(C.byref(node), parent, None, C.c_size_t(0), graph)
    for e, g in zip(execs, (graph, graph, parent)):
        cu.cuGraphInstantiateWithFlags(C.byref(e), g, C.c_ulonglong(0))
    for _ in range(4):  # two instances of one graph at once
        cu.cuGraphLaunch(execs[0], h[0])
        cu.cuGraphLaunch(execs[1], h[1])
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    out.zero_()
    torch.cuda.synchronize()
    cu.cuGraphLaunch(execs[2], h[0])
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    for e in execs:
        cu.cuGraphExecDestroy(e)
    cu.cuGraphDestroy(parent)
    cu.cuGraphDestroy(graph)
    s.close()


def test_streams_do_not_wait_for_each_other():
    s, u, want = _setup(3)
    st = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.zeros_like(u) for _ in st]
    late = torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(st[0]):
        torch.cuda._sleep(400_000_000)  # about 0.2 s ahead of the first call
        s.apply(u, outs[0], stream=st[0])
        late.record(st[0])
    s.apply(u, outs[1], stream=st[1])
    st[1].synchronize()
    assert not late.query()
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in outs)
    s.close()
