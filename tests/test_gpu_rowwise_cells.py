"""Cell solves over FP64 inverses row by row: one sweep from zero, whose entries are weighted sums of J_T^{-1} t_T, each
held to the sum of |J_T^{-1}||t_T| over its own rows; for t whose components, time nodes and pressures differ by orders
of magnitude or that is zero but for single entries, for small time steps, few and many cells and both directions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 1, 2, (3, 2)), (2, 1, 5, (16, 4)), (2, 2, 2, (5, 3)), (2, 2, 4, (10, 4)), (3, 0, 2, (3, 2, 2)),
         (3, 0, 2, (16, 4, 4)), (3, 1, 2, (2, 3, 2)), (3, 1, 2, (16, 4, 4)),
         (3, 0, 2, (16, 6, 5)), (3, 1, 2, (16, 6, 5))]


def _vectors(rng, n, k, dim, R):
    block = n // (k + 1)
    comp, time = np.minimum((np.arange(n) % block) // R, dim), np.arange(n) // block
    x = rng.standard_normal(n)
    out = {"normal": x, "zero": 0.0 * x}
    for s in (1e-2, 1e-6):
        out[f"cross flow {s}"] = x * np.where(comp == 0, 1.0, s)
        out[f"pressure {1 / s}"] = x * np.where(comp == dim, 1 / s, 1.0)
        out[f"velocity pressure {s}"] = x * np.where(comp == dim, s, 1.0)
        out[f"time {s}"] = x * s ** time
    out["wide"] = x * np.exp2(rng.integers(-20, 20, n))
    out["sparse"] = np.where(rng.random(n) < 0.01, x, 0.0)
    out["spikes"] = x * np.where(rng.random(n) < 0.01, 1e12, 1.0)
    out["small"] = x * 2.0**-1000
    return out


@pytest.mark.parametrize("dim,k,levels,cells", CASES)
@pytest.mark.parametrize("tau", [1e-2, 1e-5])
def test_rows(dim, k, levels, cells, tau):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, levels, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), tau=tau,
                              inv_precision="f64", omega=1.0))
    rng = np.random.default_rng(23)
    g, n, C = h.finest, h.n_dofs(), h.sizes(h.finest)["n_cells"]
    R = (n // (k + 1) - (dim + 1) * C) // dim
    block = n // (k + 1)
    comp = np.minimum((np.arange(n) % block) // R, dim)
    X = np.where(comp < dim, 0.3 * rng.standard_normal(n), 0.0)
    h.assemble_jacobian(torch.from_numpy(X).cuda())
    h.factor_cells()
    # the cells' unknowns: the columns of J in the cell's pressure rows, and the pressures
    J = h.copy_jacobian(g).tocsr()
    NV, NP = 3**dim, dim + 1
    idx = np.zeros((C, k + 1, dim * NV + NP), dtype=np.int64)
    for a in range(k + 1):
        p0 = a * block + dim * R + np.arange(C) * NP
        at = J.indptr[p0][:, None] + np.arange(dim * NV)
        assert (np.diff(J.indptr)[p0] == dim * NV).all()
        idx[:, a, : dim * NV] = J.indices[at]
        idx[:, a, dim * NV:] = p0[:, None] + np.arange(NP)
    idx = idx.reshape(C, -1)
    m = idx.shape[1]
    inv = h.copy_cell_inverses(g)
    owners = np.bincount(idx.reshape(-1), minlength=n)
    rows = rng.choice(n, min(n, 250), replace=False)
    cell, at = np.nonzero(np.isin(idx, rows))  # all owners of the sampled rows
    row, order = np.unique(idx[cell, at], return_inverse=True)
    for name, t in _vectors(rng, n, k, dim, R).items():
        tt = torch.from_numpy(t).cuda()
        for transpose in (False, True):
            d = torch.zeros_like(tt)
            h.vanka_sweep(g, tt, d, transpose=transpose)
            p = (inv[cell, :, at] if transpose else inv[cell, at]).astype(np.longdouble) * t[idx[cell]]
            ref, S = np.zeros(row.size, np.longdouble), np.zeros(row.size, np.longdouble)
            np.add.at(ref, order, p.sum(1))
            np.add.at(S, order, np.abs(p).sum(1))
            ref, S = ref / owners[row], (S / owners[row]).astype(float)
            # an FP64 chain of m terms per cell, at most 2^dim cells, the weights
            bound = (m + 2**dim + 4) * 2.0**-53 * S + 2.0**-1060
            err = np.abs(d.cpu().numpy()[row] - ref)
            assert (err <= bound).all(), (name, transpose, float((err / bound).max()))
    h.close()
