"""Workloads of the slab solver as a user's program runs them, and what one pass of each computes.

A case names an entry point ("op"), a channel mesh and the solver options. The meshes are the ones of
the test-suite and the benchmark: the 2.2 x 0.41 (2D) and 2.5 x 0.41 x 0.41 (3D) channel with or without
a block of obstacle cells, `levels` refinements of a cx x cy [x cz] level-1 grid, dG(k) in time.
"""
import math

import numpy as np
import torch

from paper_2107_10561_gb300 import Hierarchy, make_params

TAU, NU, GAMMA, OMEGA, INFLOW = 0.01, 1e-3, 35.0, 0.7, 0.3
DENSE = 20000  # systems up to this size are solved densely for exact()


def _case(name, op, dim, k, levels, cells, obstacle=True, inv="bf16", transpose=False):
    c = dict(op=op, dim=dim, k=k, levels=levels, cx=cells[0], cy=cells[1], cz=cells[2] if dim == 3 else 1,
             obstacle=obstacle, inv=inv, transpose=transpose)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one residual on the 32x8-cell dG(1) channel (a parity test, a coarse model)
        _case("defect_2d_small", "defect", 2, 1, 2, (16, 4), obstacle=False),
        # the Krylov operator of the benchmark: J x on 64x16x16 cells, dG(1), 962,208 unknowns
        _case("spmv_3d", "spmv", 3, 1, 3, (16, 4, 4)),
        # the adjoint's operator on the 256x64-cell dG(2) channel: J^T x, 536,448 unknowns
        _case("spmv_2d_transposed", "spmv", 2, 2, 5, (16, 4), transpose=True),
        # one smoothing step in plain FP64 on a ragged 3D mesh
        _case("sweep_3d_f64", "sweep", 3, 1, 2, (13, 5, 3), inv="f64"),
        # one V(2,2)-cycle in plain FP64 on five 2D levels, most of them small
        _case("vcycle_2d_f64", "vcycle", 2, 2, 5, (16, 4), inv="f64"),
        # the direct solve on the benchmark's 18,000-unknown level 1
        _case("coarse_3d", "coarse", 3, 1, 2, (16, 4, 4)),
        # the benchmark: one FGMRES solve of the 3D channel with BF16 cell inverses
        _case("solve_3d_bf16", "solve", 3, 1, 3, (16, 4, 4)),
        # a transposed solve with FP32 inverses on the 128x32-cell dG(1) channel (gradient workload)
        _case("adjoint_2d_f32", "adjoint", 2, 1, 4, (16, 4), inv="f32"),
        # one Newton step from a new linearisation point: assemble, invert the cells, solve
        _case("step_3d_bf16", "step", 3, 1, 2, (16, 4, 4)),
        # the same on a dG(0) mesh in 3D with odd cell counts
        _case("step_3d_dg0", "step", 3, 0, 2, (11, 3, 5), obstacle=False),
        # a nonlinear slab as time marching solves it: damped Newton on the 256x64-cell dG(2) channel
        _case("newton_2d_bf16", "newton", 2, 2, 5, (16, 4)),
        # 32 inflow scenarios that share one hierarchy
        _case("multi_3d_bf16", "multi", 3, 1, 2, (16, 4, 4)),
    ]


def draw(rng):
    op = rng.choice(["defect", "spmv", "spmv", "sweep", "vcycle", "coarse", "solve", "adjoint", "step", "newton",
                     "multi"])
    dim = 2 if op == "newton" else rng.choice([2, 3])
    k = rng.choice([0, 1, 2]) if dim == 2 else rng.choice([0, 1, 1])
    levels = rng.choice([2, 3, 4, 5]) if dim == 2 else 2
    # cells of the finest level, spread over their logarithm (at most the listed meshes' numbers)
    if dim == 2:
        top = {"step": 6000, "newton": 16000, "multi": 8000}.get(op, 16000)
        fine = math.exp(rng.uniform(math.log(200), math.log(top)))
        c1 = max(8.0, fine / 4 ** (levels - 1))
        cy = max(2, min(9, round(math.sqrt(c1 / rng.uniform(2.5, 5.5)))))
        cx, cz = max(3, min(24, round(c1 / cy))), 1
        while cx * cy * 4 ** (levels - 1) > 17000:
            levels -= 1
    else:
        top = 2000 if op in ("step", "multi", "solve", "adjoint", "coarse", "vcycle") else 10000
        fine = math.exp(rng.uniform(math.log(100), math.log(top)))
        c1 = max(12.0, fine / 8)
        cy, cz = rng.choice([(2, 2), (3, 2), (2, 3), (3, 3), (4, 3), (3, 5), (4, 4)])
        cx = max(2, min(26 if op in ("defect", "spmv", "sweep") else 16, round(c1 / (cy * cz))))
        if op in ("defect", "spmv", "sweep") and cx * cy * cz < 150 and rng.random() < 0.4:
            levels = 3
    inv = "f64" if op in ("sweep", "vcycle") else rng.choice(["bf16", "bf16", "f32", "f64"])
    obstacle = cx >= 4 and cy >= 3 and rng.random() < 0.6
    transpose = op in ("defect", "spmv", "sweep", "vcycle", "coarse") and rng.random() < 0.4
    return _case(None, op, dim, k, levels, (cx, cy, cz), obstacle, inv, transpose)


# ----------------------------------------------------------------------------------------------------
# meshes and inputs
# ----------------------------------------------------------------------------------------------------
def _cells1(case):
    return (case["cx"], case["cy"], case["cz"])[: case["dim"]]


def _length(case):
    return (2.2, 0.41) if case["dim"] == 2 else (2.5, 0.41, 0.41)


def _hole(case):
    if not case["obstacle"]:
        return (0,) * case["dim"], (0,) * case["dim"]
    return ((1, 1), (2, 2)) if case["dim"] == 2 else ((1, 1, 0), (2, 2, case["cz"]))


class _Mesh:
    """Numbering of one level: velocity nodes (x fastest, unused ones left out), then cell pressures."""

    def __init__(self, case, level):
        f = 2**level
        d, K = case["dim"], case["k"] + 1
        self.d, self.K = d, K
        self.cells = [c * f for c in _cells1(case)]
        self.h = np.array(_length(case)) / np.array(self.cells)
        lo, hi = _hole(case)
        xyz = np.stack(np.unravel_index(np.arange(int(np.prod(self.cells))), self.cells[::-1])[::-1], 1)
        self.removed = np.all((xyz >= np.array(lo) * f) & (xyz < np.array(hi) * f), axis=1)
        self.xyz = xyz[~self.removed]
        self.C = len(self.xyz)
        self.lat = [2 * c + 1 for c in self.cells]
        stride = np.cumprod([1] + self.lat[:-1])
        loc = np.array([[(i // 3**m) % 3 for m in range(d)] for i in range(3**d)])
        at = ((2 * self.xyz[:, None, :] + loc) * stride).sum(-1)
        used = np.zeros(int(np.prod(self.lat)), bool)
        used[at] = True
        self.node_lat = np.nonzero(used)[0]
        number = np.cumsum(used) - 1
        self.cell_nodes = number[at]
        self.R = self.node_lat.size
        self.block = d * self.R + (d + 1) * self.C
        self.N = K * self.block
        self.points = [np.unravel_index(self.node_lat, self.lat[::-1])[::-1][m] * self.h[m] / 2 for m in range(d)]


def _nnz(case, level):
    d, K = case["dim"], case["k"] + 1
    cells = [c * 2**level for c in _cells1(case)]
    full = int(np.prod(cells))
    lo, hi = _hole(case)
    active = full - int(np.prod([(b - a) * 2**level for a, b in zip(lo, hi)]))
    pairs = np.prod([8.0 * c + 1 for c in cells]) * active / full
    nodes = np.prod([2.0 * c + 1 for c in cells]) * active / full
    return (K * d) ** 2 * pairs + 2.0 * K * active * d * 3**d * (d + 1), K * (d * nodes + (d + 1) * active), active


def _linearisation(case, mesh, gen):
    """Channel profile and eight random divergence-free modes at the velocity nodes, zero pressure."""
    d, K, R = mesh.d, mesh.K, mesh.R
    L = _length(case)
    x = [torch.from_numpy(p).cuda() for p in mesh.points]
    prof = INFLOW * (4 if d == 2 else 16) * x[1] * (L[1] - x[1]) / L[1] ** 2
    if d == 3:
        prof = prof * x[2] * (L[2] - x[2]) / L[2] ** 2
    modes = torch.zeros(K, d, R, dtype=torch.float64, device="cuda")
    wave = torch.stack([torch.randint(1, 9 if m == 0 else 5, (8,), generator=gen) for m in range(d)]).tolist()
    amp = torch.randn(K, 8, 2, generator=gen, dtype=torch.float64).tolist()
    for m in range(8):
        a = [math.pi * wave[i][m] / L[i] for i in range(d)]
        s, c = [torch.sin(a[i] * x[i]) for i in range(d)], [torch.cos(a[i] * x[i]) for i in range(d)]
        for t in range(K):
            p, q = amp[t][m]
            if d == 2:
                modes[t, 0] += p * a[1] * s[0] * c[1]
                modes[t, 1] -= p * a[0] * c[0] * s[1]
            else:
                modes[t, 0] += p * a[1] * s[0] * c[1] * s[2] - q * a[2] * s[0] * s[1] * c[2]
                modes[t, 1] -= p * a[0] * c[0] * s[1] * s[2]
                modes[t, 2] += q * a[0] * c[0] * s[1] * s[2]
    modes *= 0.1 / modes.abs().max()
    modes[:, 0] += prof
    X = torch.zeros(K, mesh.block, dtype=torch.float64, device="cuda")
    X[:, : d * R] = modes.reshape(K, d * R)
    return X.reshape(-1)


def _inputs(case, seed):
    gen = torch.Generator().manual_seed(int(seed))
    fine = _Mesh(case, case["levels"] - 1)
    at = _Mesh(case, 0) if case["op"] == "coarse" else fine
    s = {"fine": fine, "at": at, "X": _linearisation(case, fine, gen)}
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    new = lambda *n: torch.randn(*n, generator=g, dtype=torch.float64, device="cuda")  # noqa: E731
    s["x"], s["r"] = new(at.N), new(at.N)
    if case["op"] == "multi":
        s["B"] = new(32, at.N)
    if case["op"] == "newton":
        s["U"] = INFLOW * (0.8 + 0.4 * float(torch.rand(1, generator=gen)))
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    lo, hi = _hole(case)
    h = Hierarchy(make_params(case["dim"], case["k"], case["levels"], _cells1(case), _length(case), lo, hi, TAU, NU,
                              GAMMA, GAMMA, case["inv"], "additive", OMEGA, 2, 2))
    op = case["op"]
    if op not in ("step", "newton"):
        h.assemble_jacobian(s["X"])
    if op in ("sweep", "vcycle", "coarse", "solve", "adjoint", "multi"):
        h.factor_cells()
    s["h"], s["case"] = h, case
    s["y"] = torch.zeros_like(s["B"] if op == "multi" else s["r"])
    if case["transpose"]:  # the first transposed product of a hierarchy lays J^T out; it is kept
        h.spmv(0 if op == "coarse" else h.finest, s["x"], s["y"], transpose=True)
    return s


def run(s):
    h, case, x, r, y = s["h"], s["case"], s["x"], s["r"], s["y"]
    op, tr = case["op"], case["transpose"]
    if op == "spmv":
        h.spmv(h.finest, x, y, transpose=tr)
        return y
    if op == "defect":
        h.defect(h.finest, r, x, y, transpose=tr)
        return y
    if op == "sweep":
        y.copy_(x)
        h.vanka_sweep(h.finest, r, y, transpose=tr)
        return y
    if op == "vcycle":
        h.vcycle(r, y, transpose=tr)
        return y
    if op == "coarse":
        h.coarse_solve(r, y, transpose=tr)
        return y
    if op == "solve":
        h.gmres_solve(r, y, rtol=1e-10)
        return y
    if op == "adjoint":
        h.gmres_solve(r, y, rtol=1e-10, transpose=True)
        return y
    if op == "step":
        h.assemble_jacobian(s["X"])
        h.factor_cells()
        h.gmres_solve(r, y, rtol=1e-10)
        return y
    if op == "newton":
        y.copy_(s["X"])
        info = h.newton_solve(y, s["U"], prev=s["X"])
        return {"X": y, "newton_iters": info["newton_iters"]}
    if op == "multi":
        h.gmres_solve_multi(s["B"], y, rtol=1e-10)
        return y
    raise ValueError(op)


def work(case):
    """J, the cell inverses and the coarse factors read once, the vectors in and out once; for a step and a
    Newton solve J and the inverses are written as well, and inverting a cell takes 2 n^3 operations."""
    op, d, K = case["op"], case["dim"], case["k"] + 1
    es = {"f64": 8, "f32": 4, "bf16": 2}[case["inv"]]
    n = K * (d * 3**d + d + 1)
    top = case["levels"] - 1
    nnz, N, C = _nnz(case, top)
    if op in ("spmv", "defect"):
        return {"bytes": 8 * nnz + (16 if op == "spmv" else 24) * N, "flops": 2 * nnz}
    if op == "sweep":
        return {"bytes": 8 * nnz + es * C * n * n + 24 * N, "flops": 2 * nnz + 2 * C * n * n}
    nnz0, N0, _ = _nnz(case, 0)
    slab = N0 / case["cx"]
    coarse = 8 * min(N0 * N0, 3 * N0 * slab)
    if op == "coarse":
        return {"bytes": coarse + 16 * N0, "flops": coarse / 4}
    allnnz = sum(_nnz(case, g)[0] for g in range(1, top + 1))
    cells = sum(_nnz(case, g)[2] for g in range(1, top + 1))
    cols = 32 if op == "multi" else 1
    once = {"bytes": 8 * allnnz + es * cells * n * n + coarse + 16 * N * cols,
            "flops": cols * (2 * allnnz + 2 * cells * n * n + coarse / 4)}
    if op in ("step", "newton"):
        once["bytes"] += 8 * (allnnz + nnz0) + es * cells * n * n + coarse
        once["flops"] += 2.0 * cells * n**3 + 6 * case["cx"] * slab**3
    return once


# ----------------------------------------------------------------------------------------------------
# the same results in 64 bits from the weak form, with torch alone
# ----------------------------------------------------------------------------------------------------
def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (x + 1) / 2, w / 2


def _time(k):
    c = np.zeros(k + 2)
    c[k], c[k + 1] = 1.0, -1.0
    nodes = np.sort(np.real(np.polynomial.legendre.legroots(c)))
    nodes[-1] = 1.0
    nodes = (nodes + 1) / 2
    basis = [np.poly1d(np.poly(np.delete(nodes, a)) / np.prod(nodes[a] - np.delete(nodes, a))) for a in range(k + 1)]
    s, w = _gauss(k + 3)
    v = np.array([b(s) for b in basis])
    dv = np.array([b.deriv()(s) * np.ones_like(s) for b in basis])
    v0 = np.array([b(0.0) for b in basis])
    return (TAU * np.einsum("q,aq,bq->ab", w, v, v), np.einsum("q,aq,bq->ab", w, v, dv) + np.outer(v0, v0),
            TAU * np.einsum("q,aq,bq,cq->abc", w, v, v, v))


def _shape(X):
    """Q2 values and gradients and Legendre P1 values at reference points X [q, d]."""
    d = X.shape[1]
    val = np.stack([2 * (X - 0.5) * (X - 1), -4 * X * (X - 1), 2 * X * (X - 0.5)])
    der = np.stack([4 * X - 3, -8 * X + 4, 4 * X - 1])
    phi, grad = np.ones((len(X), 3**d)), np.ones((len(X), 3**d, d))
    for i in range(3**d):
        for m in range(d):
            j = (i // 3**m) % 3
            phi[:, i] *= val[j, :, m]
            for mm in range(d):
                grad[:, i, mm] *= (der if mm == m else val)[j, :, m]
    return phi, grad, np.concatenate([np.ones((len(X), 1)), math.sqrt(3.0) * (2 * X - 1)], 1)


def _grid(d):
    x, w = _gauss(4)
    X = np.stack([g.ravel() for g in np.meshgrid(*[x] * d, indexing="ij")], 1)
    W = np.prod(np.stack([g.ravel() for g in np.meshgrid(*[w] * d, indexing="ij")]), 0)
    return X, W


class _System:
    """Element matrices of the slab Jacobian on one level at the linearisation point X of the finest."""

    def __init__(self, case, mesh, fine, X):
        d, K = mesh.d, mesh.K
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.mesh = mesh
        Mt, D, T = _time(case["k"])
        h, vol, hT = mesh.h, float(np.prod(mesh.h)), float(np.sqrt((mesh.h**2).sum()))
        Xq, W = _grid(d)
        phi, grad, xi = _shape(Xq)
        grad = grad / h
        nv, npr = 3**d, d + 1
        mass = vol * np.einsum("q,qi,qj->ij", W, phi, phi)
        stiff = vol * np.einsum("q,qim,qjm->ij", W, grad, grad)
        div = vol * np.einsum("q,qa,qjm->maj", W, xi, grad)
        A = np.zeros((1 + 2 * d, d, d, nv, nv))  # volume part, then each Dirichlet face's
        Bc, Br = np.zeros((1 + 2 * d, d, nv, npr)), np.zeros((1 + 2 * d, d, npr, nv))
        for c in range(d):
            A[0, c, c] = NU * stiff
            Bc[0, c], Br[0, c] = -div[c].T, div[c]
        Xf, Wf = _grid(d - 1)
        for f in range(2 * d):
            m, nrm = f // 2, 2.0 * (f % 2) - 1
            pf, gf, xf = _shape(np.insert(Xf, m, float(f % 2), axis=1))
            area = vol / h[m]
            S = area * np.einsum("q,qi,qj->ij", Wf, pf, pf)
            G = area * np.einsum("q,qi,qj->ij", Wf, pf, nrm * gf[:, :, m] / h[m])
            P = area * np.einsum("q,qa,qi->ai", Wf, xf, pf)
            for c in range(d):
                A[1 + f, c, c] = NU * (GAMMA / hT * S - G - G.T)
            A[1 + f, m, m] += GAMMA / hT * S
            Bc[1 + f, m], Br[1 + f, m] = nrm * P.T, -nrm * P
        mask = np.ones((mesh.C, 1 + 2 * d))
        gone = mesh.removed.reshape(mesh.cells[::-1])
        for f in range(2 * d):
            nb = mesh.xyz.copy()
            nb[:, f // 2] += 2 * (f % 2) - 1
            out = (nb < 0).any(1) | (nb >= np.array(mesh.cells)).any(1)
            inner = gone[tuple(np.clip(nb, 0, np.array(mesh.cells) - 1).T[::-1])] & ~out
            mask[:, 1 + f] = inner | (out & (f != 1))  # face 1 (x = L) is the outflow
        self.A, self.Bc, self.Br, self.mask, self.mass = t(A), t(Bc), t(Br), t(mask), t(mass)
        self.Mt, self.D, self.T = Mt, D, t(T)
        self.phi, self.grad, self.Wphi = t(phi), t(grad), t(vol * W[:, None] * phi)
        # nodal velocities: this level's nodes are nodes of the finest level
        f = fine.cells[0] // mesh.cells[0]
        co = np.unravel_index(mesh.node_lat, mesh.lat[::-1])[::-1]
        at = np.searchsorted(fine.node_lat, sum(c * f * s for c, s in zip(co, np.cumprod([1] + fine.lat[:-1]))))
        self.w = X.reshape(K, fine.block)[:, : d * fine.R].reshape(K, d, fine.R)[:, :, t(at)]
        nodes, C = mesh.cell_nodes, np.arange(mesh.C)[:, None]
        self.idx = t(np.concatenate([np.concatenate(
            [a * mesh.block + c * mesh.R + nodes for c in range(d)]
            + [a * mesh.block + d * mesh.R + C * npr + np.arange(npr)], 1) for a in range(K)], 1))
        self.nodes = t(nodes)

    def element(self, cells):
        d, K, nv, npr = self.mesh.d, self.mesh.K, 3**self.mesh.d, self.mesh.d + 1
        nt, mask = d * nv + npr, self.mask[cells]
        w = self.w[:, :, self.nodes[cells]]  # [K, d, c, nv]
        wq = torch.einsum("qs,klcs->ckql", self.phi, w)
        gw = torch.einsum("qsm,klcs->ckqlm", self.grad, w)
        adv = torch.einsum("ckqm,qjm->ckqj", wq, self.grad)
        Nv = torch.einsum("qi,qj,ckqlm->cklmij", self.Wphi, self.phi, gw)
        T1 = torch.einsum("qi,ckqj->ckij", self.Wphi, adv)
        for c in range(d):
            Nv[:, :, c, c] += T1
        A = torch.einsum("cf,flmij->clmij", mask, self.A)
        Bc = torch.einsum("cf,flia->clia", mask, self.Bc)
        Br = torch.einsum("cf,fmaj->cmaj", mask, self.Br)
        E = torch.zeros(len(mask), K * nt, K * nt, dtype=torch.float64, device="cuda")
        for a in range(K):
            for b in range(K):
                blk = self.Mt[a, b] * A + torch.einsum("k,cklmij->clmij", self.T[a, b], Nv)
                for c in range(d):
                    blk[:, c, c] += self.D[a, b] * self.mass
                e = E[:, a * nt:(a + 1) * nt, b * nt:(b + 1) * nt]
                e[:, : d * nv, : d * nv] = blk.permute(0, 1, 3, 2, 4).reshape(-1, d * nv, d * nv)
                e[:, : d * nv, d * nv:] = self.Mt[a, b] * Bc.reshape(-1, d * nv, npr)
                e[:, d * nv:, : d * nv] = self.Mt[a, b] * Br.permute(0, 2, 1, 3).reshape(-1, npr, d * nv)
        return E

    def chunks(self):
        for s in range(0, self.mesh.C, 256):
            yield torch.arange(s, min(s + 256, self.mesh.C), device="cuda")

    def apply(self, x, transpose):
        y = torch.zeros_like(x)
        for c in self.chunks():
            E = self.element(c)
            y.index_add_(0, self.idx[c].reshape(-1),
                         torch.einsum("cji,cj->ci" if transpose else "cij,cj->ci", E, x[self.idx[c]]).reshape(-1))
        return y

    def dense(self):
        N = self.mesh.N
        J = torch.zeros(N * N, dtype=torch.float64, device="cuda")
        for c in self.chunks():
            i = self.idx[c]
            J.index_add_(0, (i[:, :, None] * N + i[:, None, :]).reshape(-1), self.element(c).reshape(-1))
        return J.reshape(N, N)


def exact(case, seed):
    op, tr = case["op"], case["transpose"] or case["op"] == "adjoint"
    if op in ("vcycle", "newton"):
        return None
    s = _inputs(case, seed)
    if op not in ("spmv", "defect") and s["at"].N > DENSE:
        return None
    system = _System(case, s["at"], s["fine"], s["X"])
    if op == "spmv":
        return system.apply(s["x"], tr)
    if op == "defect":
        return s["r"] - system.apply(s["x"], tr)
    J = system.dense()
    J = J.T.contiguous() if tr else J
    if op == "sweep":
        t = s["r"] - J @ s["x"]
        step, count = torch.zeros_like(t), torch.zeros_like(t)
        for c in system.chunks():
            i = system.idx[c]
            y = torch.linalg.solve(J[i[:, :, None], i[:, None, :]], t[i].unsqueeze(-1))
            step.index_add_(0, i.reshape(-1), y.reshape(-1))
            count.index_add_(0, i.reshape(-1), torch.ones_like(y).reshape(-1))
        return s["x"] + OMEGA * step / count
    if op == "multi":
        return torch.linalg.solve(J, s["B"].T).T.contiguous()
    return torch.linalg.solve(J, s["r"].unsqueeze(-1)).squeeze(-1)
