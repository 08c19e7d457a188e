"""The 32-column product with J row by row: with R = J D formed in extended precision a sweep changes D by the rounding of
R - J D only. Every entry is held to |J_T^{-1}| times what FP64 sums may lose in the rows of its own cells, for D whose
components, time nodes and pressures differ by orders of magnitude and small time steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 0, (3, 2)), (2, 1, (4, 3)), (2, 2, (5, 3)), (3, 0, (3, 2, 2)), (3, 1, (2, 3, 2))]


def _columns(rng, n, k, dim, R, h, tau):
    block = n // (k + 1)
    comp, time = np.minimum((np.arange(n) % block) // R, dim), np.arange(n) // block
    d = rng.standard_normal((32, n))
    for o in (0, 16):
        for i, s in enumerate((1e-2, 1e-6)):
            d[o + 1 + 5 * i] *= np.where(comp == 0, 1.0, s)
            d[o + 2 + 5 * i] *= np.where(comp == dim, 1 / s, 1.0)
            d[o + 3 + 5 * i] *= np.where(comp == dim, s, 1.0)
            d[o + 4 + 5 * i] *= s ** time
            d[o + 5 + 5 * i] *= np.where(comp == dim, h / tau, 1.0)
        d[o + 11] *= np.exp2(-60.0 * np.arange(n) / n)
        d[o + 12] *= np.exp2(rng.integers(-20, 20, n))
        d[o + 13] *= rng.random(n) < 0.02
        d[o + 14] *= np.where(rng.random(n) < 0.01, 1e12, 1.0)
        d[o + 15] = 0.0
    return d


@pytest.mark.parametrize("dim,k,cells", CASES)
@pytest.mark.parametrize("tau", [1e-2, 1e-5])
@pytest.mark.parametrize("rest", [False, True])
def test_rows(dim, k, cells, tau, rest):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    length = (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41)
    h = Hierarchy(make_params(dim, k, 2, cells, length, tau=tau, inv_precision="f64", omega=1.0))
    rng = np.random.default_rng(29)
    g, n, C = h.finest, h.n_dofs(), h.sizes(h.finest)["n_cells"]
    block = n // (k + 1)
    R = (block - (dim + 1) * C) // dim
    vel = (np.arange(n) % block) < dim * R
    h.assemble_jacobian(torch.from_numpy(np.where(vel, 0.0 if rest else 0.3 * rng.standard_normal(n), 0.0)).cuda())
    h.factor_cells()
    J = h.copy_jacobian(g).tocsr()
    JT = J.T.tocsr()
    NV, NP = 3**dim, dim + 1
    idx = np.zeros((C, k + 1, dim * NV + NP), dtype=np.int64)
    for a in range(k + 1):
        p0 = a * block + dim * R + np.arange(C) * NP
        idx[:, a, : dim * NV] = J.indices[J.indptr[p0][:, None] + np.arange(dim * NV)]
        idx[:, a, dim * NV:] = p0[:, None] + np.arange(NP)
    idx = idx.reshape(C, -1)
    inv = np.abs(h.copy_cell_inverses(g))
    owners = np.bincount(idx.reshape(-1), minlength=n)
    D = _columns(rng, n, k, dim, R, length[0] / (2 * cells[0]), tau)
    Rhs, lost = np.zeros_like(D), np.zeros_like(D)
    for c in range(32):
        A = JT if c >= 16 else J
        p = A.data.astype(np.longdouble) * D[c][A.indices]
        Rhs[c] = np.add.reduceat(p, A.indptr[:-1]).astype(float)
        S = np.add.reduceat(np.abs(p), A.indptr[:-1]).astype(float)
        # an FP64 chain of m terms, the rounding of R, of R - J D
        lost[c] = (np.diff(A.indptr) + 4) * 2.0**-53 * S
    Dg, Rg = torch.from_numpy(D).cuda(), torch.from_numpy(Rhs).cuda()
    f, a = Dg[:16].clone(), Dg[16:].clone()
    h.vanka_sweep_fused(g, Rg[:16].contiguous(), f, Rg[16:].contiguous(), a)
    out = torch.cat([f, a]).cpu().numpy()
    multi = Dg.clone()
    h.vanka_sweep_multi(g, Rg, multi)
    multi = multi.cpu().numpy()
    for c in range(32):
        bound = np.zeros(n)
        amp = np.einsum("cji,cj->ci" if c >= 16 else "cij,cj->ci", inv, lost[c][idx])
        np.add.at(bound, idx.reshape(-1), amp.reshape(-1))
        bound = bound / owners * (1 + 1e-9) + 2.0**-52 * np.abs(D[c]) + 2.0**-1060
        assert (np.abs(out[c] - D[c]) <= bound).all(), (c, float((np.abs(out[c] - D[c]) / bound).max()))
        if c < 16:
            assert (np.abs(multi[c] - D[c]) <= bound).all(), (c, float((np.abs(multi[c] - D[c]) / bound).max()))
    h.close()
