"""Coarse factorisation on the tensor cores: the direct solve against a sparse LU of the same matrix over
slab sizes at the edges of the kernels (one 32-column panel, one panel of several column blocks, blocked
inverse with full and partial last panels, product tiles with remainders)."""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

pytestmark = pytest.mark.gpu

# (dim, k, level-1 cells, length): rows per x-slab from 17 to about 1,400; condition numbers up to 2e6
MESHES = [
    (2, 0, (3, 1), (2.2, 0.41)),
    (2, 0, (4, 3), (2.2, 0.41)),
    (2, 1, (3, 3), (2.2, 0.41)),
    (2, 2, (2, 5), (2.2, 0.41)),
    (2, 1, (5, 9), (2.2, 0.41)),
    (3, 0, (2, 2, 1), (2.5, 0.41, 0.41)),
    (3, 0, (3, 3, 3), (2.5, 0.41, 0.41)),
    (3, 1, (2, 3, 4), (2.5, 0.41, 0.41)),
    (3, 1, (8, 4, 5), (2.5, 0.41, 0.41)),
]


@pytest.mark.parametrize("dim,k,cells,length", MESHES)
@pytest.mark.parametrize("transpose", [False, True])
def test_coarse_solve_over_block_sizes(dim, k, cells, length, transpose):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, 2, cells, length, inv_precision="f64"))
    rng = np.random.default_rng(5)
    X = torch.from_numpy(0.1 * rng.standard_normal(h.n_dofs())).cuda()
    h.assemble_jacobian(X)
    h.factor_cells()
    n = h.n_dofs(0)
    r = rng.standard_normal(n)
    d = torch.empty(n, dtype=torch.float64, device="cuda")
    h.coarse_solve(torch.from_numpy(r).cuda(), d, transpose=transpose)
    J = h.copy_jacobian(0).tocsc()
    expect = spla.splu(J.T.tocsc() if transpose else J).solve(r)
    # an explicit inverse is off by eps x cond x a growth factor (2e-16 x 2e6 x 100 at most on these
    # meshes, far less in practice); 1e-10 as in the other coarse-solve tests
    assert np.abs(d.cpu().numpy() - expect).max() <= 1e-10 * max(1.0, np.abs(expect).max())
    h.close()
