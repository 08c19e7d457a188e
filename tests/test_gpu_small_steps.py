"""Inverses and direct solves over time steps from 1e-2 down to 1e-8, where pressures and velocities are of very different
size: the cell inverses' residuals row by row and the coarse solve's, against the same in FP64 on the host."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

pytestmark = pytest.mark.gpu


def cell_indices(h, J, dim, k):
    n, C = h.n_dofs(), h.sizes(1)["n_cells"]
    block = n // (k + 1)
    R = (block - (dim + 1) * C) // dim
    NV, NP = 3**dim, dim + 1
    idx = np.zeros((C, k + 1, dim * NV + NP), int)
    for a in range(k + 1):
        p0 = a * block + dim * R + np.arange(C) * NP
        idx[:, a, : dim * NV] = J.indices[J.indptr[p0][:, None] + np.arange(dim * NV)]
        idx[:, a, dim * NV:] = p0[:, None] + np.arange(NP)
    return idx.reshape(C, -1)


def residual(A, B):  # of A B = I, relative to |A||B|
    E = np.abs(A.astype(np.longdouble) @ B.astype(np.longdouble) - np.eye(len(A)))
    return float((E / (np.abs(A) @ np.abs(B))).max())

@pytest.mark.parametrize("dim,k,cells", [(2, 1, (4, 3)), (2, 2, (4, 3)), (3, 0, (3, 2, 2)), (3, 1, (3, 2, 2)), (3, 0, (12, 5, 5))])
@pytest.mark.parametrize("tau", [1e-2, 1e-4, 1e-6, 1e-8])
def test_inverses(dim, k, cells, tau):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, 2, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), tau=tau, inv_precision="f64"))
    rng = np.random.default_rng(1)
    h.assemble_jacobian(torch.from_numpy(0.1 * rng.standard_normal(h.n_dofs())).cuda())
    h.factor_cells()
    J, C = h.copy_jacobian(1).tocsr(), h.sizes(1)["n_cells"]
    idx = cell_indices(h, J, dim, k)
    inv = h.copy_cell_inverses(1)
    for c in range(0, C, max(1, C // 6)):
        A = J[idx[c]][:, idx[c]].toarray()
        # a backward stable inverse of the same matrix: Gauss-Jordan may lose a growth factor more
        assert residual(A, inv[c]) <= 50 * residual(A, np.linalg.inv(A)) + 1e-14, c
    J0 = h.copy_jacobian(0).tocsc()
    r = rng.standard_normal(h.n_dofs(0))
    d = torch.empty(h.n_dofs(0), dtype=torch.float64, device="cuda")
    for transpose in (False, True):
        A = J0.T.tocsc() if transpose else J0
        h.coarse_solve(torch.from_numpy(r).cuda(), d, transpose=transpose)
        # the same by an explicit inverse, as the small coarse levels' solves are
        ref = np.linalg.inv(A.toarray()) @ r if A.shape[0] < 3000 else spla.splu(A).solve(r)
        back = lambda x: float((np.abs(A @ x - r) / (abs(A) @ np.abs(x) + np.abs(r))).max())
        assert back(d.cpu().numpy()) <= 100 * back(ref) + 1e-12, transpose
    h.close()


@pytest.mark.parametrize("cells", [(3, 2, 2), (5, 3, 2)])
def test_as_exact_as_fp64_sums(cells):
    """One time node in 3D, where pivots grow least: the roundings of n sums in FP64 add up to about sqrt(n) 2^-53."""
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(3, 0, 2, cells, (2.5, 0.41, 0.41), tau=1e-2, inv_precision="f64"))
    rng = np.random.default_rng(1)
    h.assemble_jacobian(torch.from_numpy(0.1 * rng.standard_normal(h.n_dofs())).cuda())
    h.factor_cells()
    J = h.copy_jacobian(1).tocsr()
    idx, inv = cell_indices(h, J, 3, 0), h.copy_cell_inverses(1)
    for c in range(0, len(idx), 7):
        assert residual(J[idx[c]][:, idx[c]].toarray(), inv[c]) <= 4 * 85**0.5 * 2.0**-53, c
    h.close()
