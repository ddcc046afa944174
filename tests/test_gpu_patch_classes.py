"""Patch solves of the SIMT kernel for every kind of patch: one to seven elements
an axis (both ends on the boundary, next to it, between two such elements,
symmetric and not), every degree, FP64 and FP32, with few sources (one patch per
block) and many, against dense solves of the oracle's matrix restricted to the
patch. Tolerances as in test_gpu_parity.py: 1e-11 (FP64) and 1e-4 (FP32) of the
result's largest entry. A source's patches do not depend on the batch."""

import itertools

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _patch_nodes(m, pos):
    """Element-blocked index of every node of the patch of the element at pos, -1 outside the domain, x fastest."""
    lex = np.empty(m.Nq, dtype=np.int64)
    lex[oracle.dg_oracle.lex_of_eb(m)] = np.arange(m.Nq)
    ax = []
    for d in range(3):
        lo = pos[d] * m.n1 - (1 if pos[d] > 0 else 0)
        hi = (pos[d] + 1) * m.n1 + (1 if pos[d] < m.n[d] - 1 else 0)
        i = lo + np.arange(m.n1 + 2)
        ax.append(np.where(i < hi, i, -1))
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    return np.where((x >= 0) & (y >= 0) & (z >= 0), lex[x + m.L[0] * (y + m.L[1] * z)], -1).ravel()


@pytest.mark.parametrize("n,p", [((6, 6, 2), 1), ((7, 3, 1), 2), ((1, 5, 3), 3), ((4, 2, 6), 4), ((3, 1, 4), 5),
                                 ((2, 5, 1), 6), ((3, 2, 1), 7), ((1, 3, 2), 8), ((5, 1, 1), 8)])
@pytest.mark.parametrize("fp32", [False, True])
def test_patch_solves_by_class(n, p, fp32):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21213_gb300 import build, dgx

    build.build()
    lo, hi = [-2.0, -1.0, 0.5], [2.0, 1.5, 2.0]
    m = oracle.Mesh(lo, hi, n, p)
    dt = torch.float32 if fp32 else torch.float64
    # the tensor-core kernel has its own tests: off here, so that FP32 runs the SIMT kernel at every degree
    s = dgx.PoissonSolver(lo, hi, n, p, precision=dgx.DG_PREC_MIXED if fp32 else dgx.DG_PREC_FP64, tc_smoother=0)
    assert s.info.levels > 1
    B = 1 + 2 * 152 * 64 // m.E  # enough for several patches per block at every degree
    g = torch.Generator(device="cuda").manual_seed(3)
    r = torch.randn(B, m.Nq, generator=g, device="cuda", dtype=dt)
    zp = s.patch_solves(r)
    A = oracle.assemble_kron(m).tocsr()
    for k in (0, B - 1):
        one = s.patch_solves(r[k:k + 1].contiguous())
        assert torch.equal(one[0], zp[k])
        got, rk = zp[k].double().cpu().numpy(), r[k].double().cpu().numpy()
        for e, (ez, ey, ex) in enumerate(itertools.product(range(n[2]), range(n[1]), range(n[0]))):
            if e % max(1, m.E // 12):
                continue
            idx = _patch_nodes(m, (ex, ey, ez))
            inside = idx >= 0
            ref = np.zeros(idx.size)
            ref[inside] = np.linalg.solve(A[idx[inside]][:, idx[inside]].toarray(), rk[idx[inside]])
            err = np.abs(got[e] - ref).max() / np.abs(ref).max()
            assert err <= (1e-4 if fp32 else 1e-11), (e, err)
    s.close()
