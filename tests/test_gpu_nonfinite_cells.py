"""A linearisation point with one entry that is not a number: the cell inversion names a cell and the next good
point gives the inverses of a fresh hierarchy, over blocks of four and of eight warps per cell, in shared memory
and in scratch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,k,cells", [(2, 0, (5, 3)), (2, 1, (9, 4)), (2, 2, (9, 4)), (3, 0, (3, 2, 2)), (3, 1, (3, 2, 2))])
@pytest.mark.parametrize("entry", [np.nan, np.inf])
def test_one_bad_entry(dim, k, cells, entry):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, _lib, make_params
    p = make_params(dim, k, 2, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), inv_precision="f64")
    h, fresh = Hierarchy(p), Hierarchy(p)
    rng = np.random.default_rng(12)
    X = torch.from_numpy(0.3 * rng.standard_normal(h.n_dofs())).cuda()
    R = (h.n_dofs() // (k + 1) - (dim + 1) * h.sizes(h.finest)["n_cells"]) // dim
    for at in rng.choice(R, 3, replace=False):
        bad = X.clone()
        bad[int(at)] = entry
        h.assemble_jacobian(bad)
        with pytest.raises(_lib.StmError) as e:
            h.factor_cells()
        assert e.value.status == _lib.STM_ERR_SINGULAR_CELL and e.value.bad_level == 1 and e.value.bad_cell >= 0
    for q in (h, fresh):
        q.assemble_jacobian(X)
        q.factor_cells()
    assert np.array_equal(h.copy_cell_inverses(1), fresh.copy_cell_inverses(1))
    h.close()
    fresh.close()
