"""Cases for timing the library through its public entry points.

Every case is work that a Hartree-Fock or Kohn-Sham program gives this library:
whole exchange builds and operator actions (tiny to 2.1 M nodes, one system and
several, FP64 and mixed precision, uniform meshes and an octree), and the single
kernels that such a program or its own solver calls (the SIPDG operator, the
Schwarz smoother, the initial-guess network forward and backward).

Mixed-precision solves run to a residual of 1e-12, as the parity tests run
them: the potentials are then those of the discrete problem to about 1e-9 (a
residual of 1e-8 leaves 5e-6 in the energies of the largest mesh), and an
iteration does the same work whatever residual it is asked for.

`exact` gives the same outputs in 64 bits from plain torch: the discrete
problems are solved directly by fast diagonalisation of the Kronecker sum, with
none of the library's code.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_21213_gb300 import dgx, inputs

BOX = 12.0  # half width of the box, bohr
PRECISIONS = {"fp64": dgx.DG_PREC_FP64, "mixed": dgx.DG_PREC_MIXED}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # two s-Gaussians on 64 elements: a test-sized molecule, where launches and latency count
        {"name": "build_tiny_fp64", "kind": "build", "system": "tiny", "nx": 4, "ny": 4, "nz": 4, "p": 4, "N": 2,
         "precision": "fp64", "rtol": 1e-10},
        # the ten-atom chain, every occupied pair: one Fock exchange build of an SCF step
        {"name": "build_chain10_mixed", "kind": "build", "system": "chain", "nx": 8, "ny": 8, "nz": 8, "p": 6,
         "N": 10, "precision": "mixed", "rtol": 1e-12},
        # the same build with every step in FP64 (reference energies)
        {"name": "build_chain10_fp64", "kind": "build", "system": "chain", "nx": 8, "ny": 8, "nz": 8, "p": 6,
         "N": 10, "precision": "fp64", "rtol": 1e-10},
        # one library batch of the 16^3, p = 7, 64-orbital build (a rank's share of a large system)
        {"name": "range_16c_p7_mixed", "kind": "range", "system": "random", "nx": 16, "ny": 16, "nz": 16, "p": 7,
         "N": 64, "S": 42, "precision": "mixed", "rtol": 1e-12},
        # Hartree and exchange action on trial functions (an eigensolver's step), uneven box, odd degree
        {"name": "jk_uneven_mixed", "kind": "jk", "system": "random", "nx": 6, "ny": 10, "nz": 8, "p": 5, "N": 4,
         "m": 5, "precision": "mixed", "rtol": 1e-12},
        # potentials of a few densities in FP64 at the highest degree, uneven box
        {"name": "solve_p8_fp64", "kind": "solve", "system": "random", "nx": 6, "ny": 8, "nz": 4, "p": 8, "B": 5,
         "precision": "fp64", "rtol": 1e-10},
        # several molecules of uneven size in one call
        {"name": "multi5_mixed", "kind": "multi", "systems": "8.6.8,6.7.6,4.8.12,6.5.10,4.4.3", "precision": "mixed",
         "rtol": 1e-12},
        # potentials on a density-refined octree (hanging faces)
        {"name": "octree_mixed", "kind": "octree", "n": 8, "p": 6, "max_level": 2, "B": 8, "precision": "mixed",
         "rtol": 1e-12},
        # the operator alone on one library batch, as an outer Krylov solver applies it
        {"name": "operator_16c_p7_fp32", "kind": "operator", "nx": 16, "ny": 16, "nz": 16, "p": 7, "B": 42,
         "dtype": "fp32"},
        # the smoother alone on one library batch, as an outer preconditioner applies it
        {"name": "smoother_16c_p7_fp32", "kind": "smoother", "nx": 16, "ny": 16, "nz": 16, "p": 7, "B": 42,
         "dtype": "fp32"},
        # the smoother on a few fields of a small odd-sized mesh in FP64
        {"name": "smoother_odd_fp64", "kind": "smoother", "nx": 5, "ny": 7, "nz": 3, "p": 5, "B": 3, "dtype": "fp64"},
        # network of the initial guess, forward and backward on one training batch of four sources
        {"name": "network_train_p7", "kind": "network", "p": 7, "elements": 16384},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "range", "jk", "solve", "multi", "octree", "operator", "operator", "smoother",
                       "smoother", "network"])
    prec = rng.choice(["fp64", "mixed"])
    rtol = {"fp64": 1e-10, "mixed": 1e-12}[prec]
    p = rng.randint(4, 8)
    n = [rng.randint(3, 10) for _ in range(3)]
    if rng.random() < 0.6:  # sizes that coarsen
        n = [v - v % 2 + (2 if v < 4 else 0) for v in n]
    # odd counts stop the coarsening: what is left has to be a size that a direct coarsest solve suits
    while any(v % 2 for v in n) and n[0] * n[1] * n[2] > 140:
        n[n.index(max(n))] -= 1
    nodes = n[0] * n[1] * n[2] * (p + 1) ** 3
    mesh = {"nx": n[0], "ny": n[1], "nz": n[2], "p": p}
    if kind in ("operator", "smoother"):
        # small odd meshes to 16^3 elements, one field to one library batch
        if rng.random() < 0.5:
            k = rng.choice([8, 10, 12, 16])
            mesh.update(nx=k, ny=k, nz=rng.choice([k, 8, 12]))
            nodes = mesh["nx"] * mesh["ny"] * mesh["nz"] * (p + 1) ** 3
        top = max(1, min(64, int(80e6 / nodes)))
        return {"kind": kind, **mesh, "B": _log_int(rng, 1, top), "dtype": rng.choice(["fp32", "fp64"])}
    if kind == "network":
        return {"kind": kind, "p": rng.randint(4, 7), "elements": _log_int(rng, 200, 16384)}
    if kind == "octree":
        return {"kind": kind, "n": rng.choice([4, 6, 8]), "p": rng.randint(4, 6), "max_level": rng.randint(1, 2),
                "B": _log_int(rng, 1, 12), "precision": "mixed", "rtol": 1e-12}
    if kind == "multi":
        systems = [(rng.choice([4, 6, 8]), rng.randint(4, 8), rng.randint(2, 6)) for _ in range(rng.randint(2, 5))]
        return {"kind": kind, "systems": ",".join("%d.%d.%d" % s for s in systems), "precision": "mixed",
                "rtol": 1e-12}
    # whole solves: the sources are chosen so that a case costs no more than the chain's FP64 build
    most = max(2, min(60, int((9e6 if prec == "fp64" else 60e6) / nodes)))
    if kind == "build":
        N = min(10, int((math.sqrt(8 * most + 1) - 1) / 2))
        return {"kind": kind, "system": rng.choice(["chain", "random"]), **mesh, "N": rng.randint(1, max(1, N)),
                "precision": prec, "rtol": rtol}
    if kind == "range":
        return {"kind": kind, "system": "random", **mesh, "N": rng.randint(4, 32), "S": min(10, _log_int(rng, 1, most)),
                "precision": prec, "rtol": rtol}
    if kind == "jk":
        N = rng.randint(1, 6)
        return {"kind": kind, "system": "random", **mesh, "N": N, "m": rng.randint(1, max(1, min(8, most // N))),
                "precision": prec, "rtol": rtol}
    return {"kind": "solve", "system": "random", **mesh, "B": _log_int(rng, 1, most), "precision": prec, "rtol": rtol}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _mesh(case):
    half = 8.0 if case.get("system") == "tiny" else BOX
    return (-half,) * 3, (half,) * 3, (case["nx"], case["ny"], case["nz"]), case["p"]


def _system(kind, lo, hi, n, p, N, seed):
    mesh = inputs.MeshSpec(lo, hi, n, p)
    if kind == "tiny":
        rng = np.random.default_rng(seed)
        spec = inputs.tiny_system()
        spec.atoms = spec.atoms + rng.uniform(-0.3, 0.3, size=spec.atoms.shape)
        spec.exponents = np.exp(rng.uniform(math.log(0.8), math.log(1.25), size=2))
        return spec
    if kind == "chain":
        atoms = np.array([[-6.3 + 1.4 * k, 0.0, 0.0] for k in range(10)])
    else:
        atoms = inputs.random_system(seed=seed, n=2, p=1, n_orb=1, n_atoms=N // 2 + 1).atoms
    return inputs.gto_system(mesh, atoms, N, seed)


def _orbitals(spec, xyz, w):
    x, ww = (torch.as_tensor(v, device="cuda", dtype=torch.float64) for v in (xyz, w))
    if spec.kind == "gto":
        return inputs.orbitals_torch(spec, x, ww)
    return torch.tensor(inputs.orbitals(spec, np.asarray(xyz), np.asarray(w)), device="cuda")


def _fields(case, seed, nodes):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(case["B"], nodes, generator=g, device="cuda",
                       dtype=torch.float32 if case["dtype"] == "fp32" else torch.float64)


def _densities(spec, xyz, w, B):
    """B sources as they come up between builds: the density, then pair densities."""
    psi = _orbitals(spec, xyz, w)
    N = psi.shape[0]
    f = [psi.square().sum(dim=0)]
    f += [psi[i] * psi[j] for i in range(N) for j in range(i, N)]
    return torch.stack(f[:B]).contiguous()


def _orbital_count(sources):
    return max(1, math.ceil((math.sqrt(8 * sources + 1) - 1) / 2))


def _octree(case, seed):
    """Root mesh, orbitals and the leaves refined by their density."""
    lo, hi, n = (-BOX,) * 3, (BOX,) * 3, (case["n"],) * 3
    spec = _system("chain", lo, hi, n, case["p"], max(4, _orbital_count(case["B"])), seed)
    # the mesh is refined for the geometry's typical density, as in an SCF run: it does not follow the seed
    typical = _system("chain", lo, hi, n, case["p"], 10, 2)

    def rho(x):
        return np.sum((typical.coeffs @ inputs.eval_primitives(typical, x)) ** 2, axis=0)

    return lo, hi, n, spec, dgx.dg_octree_refine(lo, hi, n, case["p"], rho, 1e-5, case["max_level"])


def _multi(case):
    return [tuple(int(v) for v in s.split(".")) for s in case["systems"].split(",")]


def _network(case, seed):
    """Weights near the trained ones, inputs and output gradients of one training batch."""
    g = torch.Generator().manual_seed(seed)
    scale = {"W1": 54, "b1": 0, "W2": 864, "b2": 0, "W3": 864, "b3": 0}
    prm = {k: torch.randn(shape, generator=g, dtype=torch.float64) * (math.sqrt(2.0 / scale[k]) if scale[k] else 0.05)
           for k, shape in dgx.NN_LAYOUT}
    gd = torch.Generator(device="cuda").manual_seed(seed)
    n1 = case["p"] + 1
    t = torch.linspace(-1, 1, n1, device="cuda")
    z, y, x = torch.meshgrid(t, t, t, indexing="ij")
    modes = torch.stack([torch.ones_like(x), x, y, z, x * y, y * z, z * x, x * x, y * y, z * z]).reshape(10, -1)
    c = torch.randn(case["elements"], 2, 10, generator=gd, device="cuda")
    xin = (c @ modes).transpose(1, 2).contiguous() * 0.3
    gout = torch.randn(case["elements"], n1 ** 3, 2, generator=gd, device="cuda") * 1e-3
    return prm, xin, gout


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("operator", "smoother"):
        lo, hi, n, p = _mesh(case)
        prec = PRECISIONS["mixed" if case["dtype"] == "fp32" else "fp64"]
        s = dgx.PoissonSolver(lo, hi, n, p, precision=prec)
        return {"kind": kind, "solver": s, "u": _fields(case, seed, s.Nq)}
    if kind == "network":
        prm, xin, gout = _network(case, seed)
        s = dgx.PoissonSolver((-BOX,) * 3, (BOX,) * 3, (2, 2, 2), case["p"], precision=dgx.DG_PREC_MIXED)
        dgx.dg_nn_set_params(s.h, dgx.nn_pack({k: v.numpy() for k, v in prm.items()}))
        return {"kind": kind, "solver": s, "x": xin, "gout": gout}
    if kind == "octree":
        lo, hi, n, spec, leaves = _octree(case, seed)
        s = dgx.OctreeSolver(lo, hi, n, case["p"], leaves, rtol=case["rtol"], precision=PRECISIONS[case["precision"]])
        xyz, w = s.node_coords()
        return {"kind": kind, "solver": s, "f": _densities(spec, xyz, w, case["B"])}
    if kind == "multi":
        systems = []
        for i, (n, p, N) in enumerate(_multi(case)):
            lo, hi = (-BOX,) * 3, (BOX,) * 3
            spec = _system("random", lo, hi, (n,) * 3, p, N, seed + 101 * i)
            xyz, w = dgx.dg_mesh_node_coords(lo, hi, n, p)
            systems.append((lo, hi, (n,) * 3, p, _orbitals(spec, xyz, w)))
        return {"kind": kind, "systems": systems,
                "opts": dgx.dg_default_opts(precision=PRECISIONS[case["precision"]], rtol=case["rtol"])}
    lo, hi, n, p = _mesh(case)
    s = dgx.PoissonSolver(lo, hi, n, p, precision=PRECISIONS[case["precision"]], rtol=case["rtol"])
    xyz, w = s.node_coords()
    if kind == "solve":
        spec = _system(case["system"], lo, hi, n, p, _orbital_count(case["B"]), seed)
        return {"kind": kind, "solver": s, "f": _densities(spec, xyz, w, case["B"])}
    spec = _system(case["system"], lo, hi, n, p, case["N"], seed)
    state = {"kind": kind, "solver": s, "psi": _orbitals(spec, xyz, w)}
    if kind == "range":
        state["S"] = min(case["S"], case["N"] * (case["N"] + 1) // 2 + 1)
    if kind == "jk":
        state["U"] = _trial(spec, xyz, w, case["m"], seed)
    return state


def _trial(spec, xyz, w, m, seed):
    """Trial functions of an eigensolver: other combinations of the same atoms' functions."""
    other = inputs.gto_system(spec.mesh, spec.atoms, min(m, 4 * len(spec.atoms)), seed + 17)
    u = _orbitals(other, xyz, w)
    return u.repeat(-(-m // u.shape[0]), 1)[:m].contiguous()


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _build_out(K, eh, ex, stats):
    return {"K": K, "E_H": np.float64(eh), "E_X": np.float64(ex), "self": np.array([t["self_energy"] for t in stats])}


def run(state):
    kind, s = state["kind"], state.get("solver")
    if kind == "operator":
        return s.apply(state["u"])
    if kind == "smoother":
        return s.smoother(state["u"])
    if kind == "network":
        out = dgx.dg_nn_forward(s.h, state["x"], save_act=True)
        return {"out": out, "grad": dgx.dg_nn_backward(s.h, state["x"], state["gout"])}
    if kind in ("solve", "octree"):
        v, stats = s.solve(state["f"])
        return {"v": v, "self": np.array([t["self_energy"] for t in stats])}
    if kind == "build":
        return _build_out(*s.exchange_build(state["psi"]))
    if kind == "range":
        K, eh, stats = s.exchange_build_range(state["psi"], 0, state["S"])
        return {"K": K, "E_H": np.float64(eh), "self": np.array([t["self_energy"] for t in stats])}
    if kind == "jk":
        JU, XU, stats = s.jk_apply(state["psi"], state["U"])
        return {"JU": JU, "XU": XU}
    Ks, eh, ex, stats = dgx.dg_exchange_build_multi(state["systems"], state["opts"])
    return [_build_out(K, h, x, t) for K, h, x, t in zip(Ks, eh, ex, stats)]


# ---------------------------------------------------------------------------
# work that cannot be done without
# ---------------------------------------------------------------------------
def _solve_flops(nodes, n1, sources):
    """A solve to its residual: about 6 multigrid-CG iterations, each with 8 smoothing steps (operator and
    exact patch solves) on the fine level; the coarse levels add about a seventh."""
    m = n1 + 2
    return 6.0 * 8.0 * (6 * n1 + 56 + 12.0 * m ** 4 / n1 ** 3) * 8.0 / 7.0 * nodes * sources


def work(case):
    kind = case["kind"]
    if kind == "network":
        n1 = case["p"] + 1
        per = 2.0 * 27 * (2 * 32 + 32 * 32 + 32 * 2) * n1 ** 3
        return {"bytes": case["elements"] * n1 ** 3 * 3 * 8.0 + 2 * 4 * 31170, "flops": 3 * per * case["elements"]}
    if kind == "octree":
        # leaves: the roots plus the refined chain neighbourhood (about 40 % more of them at level 2)
        nodes = case["n"] ** 3 * (1.2 if case["max_level"] == 1 else 1.4) * (case["p"] + 1) ** 3
        return {"bytes": 2 * 8.0 * nodes * case["B"], "flops": 4 * _solve_flops(nodes, case["p"] + 1, case["B"])}
    if kind == "multi":
        b = f = 0.0
        for n, p, N in _multi(case):
            nodes = n ** 3 * (p + 1) ** 3
            b += 8.0 * nodes * N + 8.0 * N * N
            f += _solve_flops(nodes, p + 1, N * (N + 1) // 2 + 1)
        return {"bytes": b, "flops": f}
    n1 = case["p"] + 1
    nodes = case["nx"] * case["ny"] * case["nz"] * n1 ** 3
    if kind in ("operator", "smoother"):
        size = 4.0 if case["dtype"] == "fp32" else 8.0
        per = 6 * n1 + 56 if kind == "operator" else 12.0 * (n1 + 2) ** 4 / n1 ** 3
        return {"bytes": 2 * size * nodes * case["B"], "flops": per * nodes * case["B"]}
    if kind == "solve":
        return {"bytes": 16.0 * nodes * case["B"], "flops": _solve_flops(nodes, n1, case["B"])}
    N = case["N"]
    if kind == "jk":
        return {"bytes": 8.0 * nodes * (N + 3 * case["m"]), "flops": _solve_flops(nodes, n1, N * case["m"] + 1)}
    sources = N * (N + 1) // 2 + 1
    if kind == "range":
        sources = min(case["S"], sources)
    return {"bytes": 8.0 * nodes * N + 8.0 * N * N, "flops": _solve_flops(nodes, n1, sources) + 2.0 * N * N * nodes}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _lagrange(x, at):
    """Values and derivatives at one point of the Lagrange basis on the nodes x."""
    k = len(x)
    val, der = np.ones(k), np.zeros(k)
    for i in range(k):
        others = [j for j in range(k) if j != i]
        val[i] = np.prod([(at - x[j]) / (x[i] - x[j]) for j in others])
        der[i] = sum(np.prod([1.0 / (x[i] - x[j])] + [(at - x[l]) / (x[i] - x[l]) for l in others if l != j])
                     for j in others)
    return val, der


class _Axis:
    """Global 1-D SIPDG matrix A, mass m, nodes x and boundary load vectors of one axis."""

    def __init__(self, lo, hi, n, p):
        xi, w = np.polynomial.legendre.leggauss(p + 1)
        h, n1 = (hi - lo) / n, p + 1
        self.n, self.n1, self.L = n, n1, n * n1
        self.x = (lo + h * (np.arange(n)[:, None] + (xi[None, :] + 1) / 2)).ravel()
        self.m = np.tile(w * h / 2, n)
        self.ends = (lo, hi)
        sigma = n1 * n1 / (0.125 * h)
        (vl, dl), (vr, dr) = _lagrange(xi, -1.0), _lagrange(xi, 1.0)
        dl, dr = dl * 2 / h, dr * 2 / h
        D = np.stack([_lagrange(xi, t)[1] for t in xi]) * 2 / h
        A = np.zeros((self.L, self.L))
        for e in range(n):
            s = slice(e * n1, e * n1 + n1)
            A[s, s] += D.T @ ((w * h / 2)[:, None] * D)
        for e in range(n + 1):  # face between elements e - 1 and e
            s = slice(max(e - 1, 0) * n1, min(e + 1, n) * n1)
            if e == 0:
                jump, avg = -vl, dl
            elif e == n:
                jump, avg = vr, dr
            else:
                jump, avg = np.concatenate([vr, -vl]), np.concatenate([dr, dl]) / 2
            A[s, s] += sigma * np.outer(jump, jump) - np.outer(jump, avg) - np.outer(avg, jump)
        self.A = A
        # load of unit Dirichlet data at either end: sigma v - d_n v
        self.load = (np.concatenate([sigma * vl + dl, np.zeros(self.L - n1)]),
                     np.concatenate([np.zeros(self.L - n1), sigma * vr - dr]))


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


class _Exact:
    """One uniform mesh in 64 bits. Fields are [B, Lz, Ly, Lx] in lexicographic order."""

    def __init__(self, lo, hi, n, p):
        self.n, self.n1 = n, p + 1
        self.ax = [_Axis(lo[d], hi[d], n[d], p) for d in range(3)]
        self.A = [_t(a.A) for a in self.ax]
        self.m = [_t(a.m) for a in self.ax]
        self.lam, self.S = [], []
        for a in self.ax:
            r = 1 / np.sqrt(a.m)
            lam, q = np.linalg.eigh(r[:, None] * a.A * r[None, :])
            self.lam.append(_t(lam))
            self.S.append(_t(r[:, None] * q))
        self.gauss = None

    def lex(self, f):
        nx, ny, nz = self.n
        k = self.n1
        return f.double().reshape(-1, nz, ny, nx, k, k, k).permute(0, 1, 4, 2, 5, 3, 6).reshape(-1, nz * k, ny * k, nx * k)

    def blocked(self, f):
        nx, ny, nz = self.n
        k = self.n1
        return f.reshape(-1, nz, k, ny, k, nx, k).permute(0, 1, 3, 5, 2, 4, 6).reshape(f.shape[0], -1)

    def weights(self):
        return self.m[2][:, None, None] * self.m[1][:, None] * self.m[0]

    def apply(self, u):
        Ax, Ay, Az = self.A
        mx, my, mz = self.m
        out = torch.einsum("ij,bzyj->bzyi", Ax, u) * (mz[:, None, None] * my[:, None])
        out += torch.einsum("ij,bzjx->bzix", Ay, u) * (mz[:, None, None] * mx)
        out += torch.einsum("ij,bjyx->biyx", Az, u) * (my[:, None] * mx)
        return out

    def smooth(self, r):
        """Sum of the exact solves on every element's patch (the element and one layer of nodes around it)."""
        idx, S, lam = [], [], []
        for a in self.ax:
            m = a.n1 + 2
            at = np.arange(a.n)[:, None] * a.n1 - 1 + np.arange(m)[None, :]
            s, l = np.zeros((a.n, m, m)), np.ones((a.n, m))
            for e in range(a.n):
                ok = np.flatnonzero((at[e] >= 0) & (at[e] < a.L))
                i = at[e][ok]
                q = 1 / np.sqrt(a.m[i])
                ev, v = np.linalg.eigh(q[:, None] * a.A[np.ix_(i, i)] * q[None, :])
                s[e][np.ix_(ok, np.arange(len(ok)))] = q[:, None] * v
                l[e, : len(ok)] = ev
            idx.append(torch.as_tensor(np.clip(at, 0, a.L - 1), device="cuda"))
            S.append(_t(s))
            lam.append(_t(l))
        den = (lam[2][:, None, None, :, None, None] + lam[1][None, :, None, None, :, None]
               + lam[0][None, None, :, None, None, :])
        iz, iy, ix = idx[2][:, None, None, :, None, None], idx[1][None, :, None, None, :, None], idx[0][None, None, :, None, None, :]
        flat = ((iz * self.ax[1].L + iy) * self.ax[0].L + ix).expand(den.shape).reshape(-1)
        out = torch.zeros_like(r)
        for b in range(r.shape[0]):  # entries outside the domain meet zero rows of S
            t = r[b].reshape(-1)[flat].reshape(den.shape)
            for k, spec in enumerate(("xiq,zyxkji->zyxkjq", "yjq,zyxkji->zyxkqi", "zkq,zyxkji->zyxqji")):
                t = torch.einsum(spec, S[k], t)
            t = t / den
            for k, spec in enumerate(("xiq,zyxkjq->zyxkji", "yjq,zyxkqi->zyxkji", "zkq,zyxqji->zyxkji")):
                t = torch.einsum(spec, S[k], t)
            out[b].reshape(-1).index_add_(0, flat, t.reshape(-1))
        return out

    def _terms(self):
        """1/r as a sum of Gaussians: the trapezoidal rule of (2/sqrt(pi)) int exp(-r^2 e^(2t) + t) dt."""
        if self.gauss is None:
            rmin = min(min(a.x[0] - a.ends[0], a.ends[1] - a.x[-1]) for a in self.ax)
            rmax = math.sqrt(sum((a.ends[1] - a.ends[0]) ** 2 for a in self.ax))
            t = np.arange(-34.0 - math.log(rmax), math.log(6.5 / rmin), 0.13)
            keep = np.exp(t) * rmax > 1e-15
            t = t[keep]
            self.gauss = (0.13 * 2 / math.sqrt(math.pi) * np.exp(t), np.exp(2 * t))
        return self.gauss

    def boundary(self, f):
        """Coulomb potential of the sources f at the face nodes: {(axis, side): [B, L_high, L_low]}."""
        c, al = self._terms()
        wf = f * self.weights()
        g = {(d, s): 0.0 for d in range(3) for s in range(2)}
        for k in range(len(c)):
            G = [_t(np.exp(-al[k] * (a.x[:, None] - a.x[None, :]) ** 2)) for a in self.ax]
            for d in range(3):
                lowered = "bzyx,sx->bszy" if d == 0 else ("bzyx,sy->bszx" if d == 1 else "bzyx,sz->bsyx")
                a = self.ax[d]
                e = _t(np.stack([np.exp(-al[k] * (a.x - x) ** 2) for x in a.ends]))
                t1, t2 = [j for j in range(3) if j != d]
                t = G[t2] @ torch.einsum(lowered, wf, e) @ G[t1]
                for s in range(2):
                    g[d, s] = g[d, s] + c[k] * t[:, s]
        return g

    def solve(self, f):
        g = self.boundary(f)
        b = 4 * math.pi * self.weights() * f
        for (d, s), v in g.items():
            l = _t(self.ax[d].load[s])
            t1, t2 = [j for j in range(3) if j != d]
            v = v * (self.m[t2][:, None] * self.m[t1])
            spec = "bzy,x->bzyx" if d == 0 else ("bzx,y->bzyx" if d == 1 else "byx,z->bzyx")
            b += torch.einsum(spec, v, l)
        Sx, Sy, Sz = self.S
        t = Sz.T @ torch.einsum("bzyx,yq->bzqx", b @ Sx, Sy).reshape(b.shape[0], b.shape[1], -1)
        t = t.reshape(b.shape) / (self.lam[2][:, None, None] + self.lam[1][:, None] + self.lam[0])
        t = (Sz @ t.reshape(b.shape[0], b.shape[1], -1)).reshape(b.shape)
        return torch.einsum("bzqx,yq->bzyx", t, Sy) @ Sx.T


def _exact_build(E, psi, sources):
    """K's contribution of the sources (0: the density, then the pairs), E_H and every source's self-energy."""
    N = psi.shape[0]
    W = E.weights()
    pairs = [(i, j) for i in range(N) for j in range(i, N)]
    acc = torch.zeros_like(psi)
    eh, self_e = 0.0, []
    for at in range(0, sources, 8):
        chunk = range(at, min(at + 8, sources))
        f = torch.stack([psi.square().sum(dim=0) if k == 0 else psi[pairs[k - 1][0]] * psi[pairs[k - 1][1]] for k in chunk])
        v = E.solve(f)
        for k, fk, vk in zip(chunk, f, v):
            self_e.append(float((W * fk * vk).sum()))
            if k == 0:
                eh = 0.5 * self_e[-1]
            else:
                i, j = pairs[k - 1]
                acc[j] += psi[i] * vk
                if i != j:
                    acc[i] += psi[j] * vk
    K = (psi * W).reshape(N, -1) @ acc.reshape(N, -1).T
    return {"K": K.cpu().numpy(), "E_H": np.float64(eh), "E_X": np.float64(-0.5 * float(K.trace())),
            "self": np.array(self_e)}


def _exact_network(prm, x, gout):
    """Output and parameter gradient of the three zero-padded 3x3x3 convolutions."""
    ne, n1 = x.shape[0], round(x.shape[1] ** (1 / 3))
    prm = {k: v.float().double().cuda().requires_grad_(True) for k, v in prm.items()}

    def conv(a, W, b):
        pad = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        y = b.expand(*a.shape[:-1], W.shape[-1])
        for z in range(3):
            for yy in range(3):
                for xx in range(3):
                    y = y + pad[:, z:z + n1, yy:yy + n1, xx:xx + n1] @ W[z, yy, xx]
        return y

    outs = []
    for at in range(0, ne, 1024):
        a = x[at:at + 1024].double().reshape(-1, n1, n1, n1, 2)
        a = torch.relu(conv(a, prm["W1"], prm["b1"]))
        a = torch.relu(conv(a, prm["W2"], prm["b2"]))
        o = conv(a, prm["W3"], prm["b3"]).reshape(a.shape[0], -1, 2)
        o.backward(gout[at:at + 1024].double())
        outs.append(o.detach())
    grad = torch.cat([prm[k].grad.reshape(-1) for k, _ in dgx.NN_LAYOUT])
    return {"out": torch.cat(outs), "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "octree":
        return None  # an independent direct solve on the octree takes minutes
    if kind == "network":
        return _exact_network(*_network(case, seed))
    if kind == "multi":
        out = []
        for i, (n, p, N) in enumerate(_multi(case)):
            lo, hi = (-BOX,) * 3, (BOX,) * 3
            E = _Exact(lo, hi, (n,) * 3, p)
            psi = _exact_orbitals(E, _system("random", lo, hi, (n,) * 3, p, N, seed + 101 * i))
            out.append(_exact_build(E, psi, N * (N + 1) // 2 + 1))
        return out
    lo, hi, n, p = _mesh(case)
    E = _Exact(lo, hi, n, p)
    if kind in ("operator", "smoother"):
        u = _fields(case, seed, n[0] * n[1] * n[2] * (p + 1) ** 3)
        step = E.apply if kind == "operator" else E.smooth
        return torch.cat([E.blocked(step(E.lex(u[k:k + 4]))) for k in range(0, u.shape[0], 4)])
    if kind == "solve":
        psi = _exact_orbitals(E, _system(case["system"], lo, hi, n, p, _orbital_count(case["B"]), seed))
        N = psi.shape[0]
        f = [psi.square().sum(dim=0)] + [psi[i] * psi[j] for i in range(N) for j in range(i, N)]
        f = torch.stack(f[: case["B"]])
        v = torch.cat([E.solve(f[k:k + 8]) for k in range(0, f.shape[0], 8)])
        return {"v": E.blocked(v), "self": (E.weights() * f * v).sum(dim=(1, 2, 3)).cpu().numpy()}
    spec = _system(case["system"], lo, hi, n, p, case["N"], seed)
    psi = _exact_orbitals(E, spec)
    N = psi.shape[0]
    if kind == "jk":
        xyz, w = _coords(E)
        U = E.lex(_trial(spec, xyz, w, case["m"], seed))
        v = E.solve(psi.square().sum(dim=0)[None])[0]
        XU = torch.zeros_like(U)
        for k in range(U.shape[0]):
            XU[k] = -(psi * E.solve(psi * U[k])).sum(dim=0)
        return {"JU": E.blocked(v * U), "XU": E.blocked(XU)}
    total = N * (N + 1) // 2 + 1
    out = _exact_build(E, psi, total if kind == "build" else min(case["S"], total))
    if kind == "range":
        del out["E_X"]
    return out


def _coords(E):
    """Coordinates and weights of the nodes, element-blocked."""
    z, y, x = torch.meshgrid(*[_t(E.ax[d].x) for d in (2, 1, 0)], indexing="ij")
    xyz = torch.stack([E.blocked(v[None])[0] for v in (x, y, z)], dim=1)
    return xyz.cpu().numpy(), E.blocked(E.weights()[None])[0].cpu().numpy()


def _exact_orbitals(E, spec):
    return E.lex(_orbitals(spec, *_coords(E)))
