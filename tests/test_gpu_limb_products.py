"""J x and b - J x on the levels whose velocity rows are two-limb integers: every number of rows per node that is
kept so, meshes with full and ragged neighbour lists, J and its transpose, and x over magnitudes that differ from
node to node, against sums in extended precision; entries that integers cannot hold against the CSR product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one, two and three time nodes in 3D, small and larger levels (8 to 32 lanes per node); 2D dG(2) from 12,000 nodes on
CASES = [(3, 0, 2, (3, 2, 2)), (3, 1, 2, (2, 3, 2)), (3, 1, 3, (14, 4, 4)), (3, 2, 2, (3, 2, 2)), (2, 2, 5, (6, 3)),
         (2, 2, 5, (10, 4))]


def _hierarchy(dim, k, levels, cells):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, levels, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41)))
    rng = np.random.default_rng(4)
    h.assemble_jacobian(torch.from_numpy(0.3 * rng.standard_normal(h.n_dofs())).cuda())
    return h, rng


def _vectors(rng, n):
    x = rng.standard_normal(n)
    return {"normal": x, "wide": x * np.exp2(rng.integers(-60, 60, n)), "decay": x * np.exp2(-200.0 * np.arange(n) / n),
            "sparse": x * (rng.random(n) < 0.01), "tiny": x * 2.0**-1010, "zero": 0.0 * x}


def _bound(A, x, rows, block, nvel, dim):
    """Per row of the nodes sampled: a value keeps 58 bits below the largest of its row, an entry of x 58 below the largest around the
    node, and the pressure columns of a node one common offset (a power of two above the largest ratio of pressure to
    velocity values in its rows, so less than 8 of it with the exponents of both): less than 2^-55 of the largest product per term, and two roundings of the sum."""
    node = {}
    for r in rows:
        a, v = divmod(r, block)
        node.setdefault((v % (nvel // dim)), []).append(r)
    out = {}
    for rr in node.values():
        pmax = vmax = xv = xp = ratio = 0.0
        for r in rr:
            s = slice(A.indptr[r], A.indptr[r + 1])
            c, v = A.indices[s], np.abs(A.data[s])
            p = c % block >= nvel
            xv, xp = max(xv, np.abs(x[c[~p]]).max()), max(xp, np.abs(x[c[p]]).max())
            ratio = max(ratio, v[p].max() / v[~p].max())
        for r in rr:
            s = slice(A.indptr[r], A.indptr[r + 1])
            v = np.abs(A.data[s][A.indices[s] % block < nvel]).max()
            out[r] = (s.stop - s.start) * 2.0**-55 * 2 * v * max(2 * xv, 8 * ratio * xp)
    return np.array([out[r] for r in rows])


@pytest.mark.parametrize("dim,k,levels,cells", CASES)
@pytest.mark.parametrize("transpose", [False, True])
def test_against_extended_precision(dim, k, levels, cells, transpose):
    import torch
    h, rng = _hierarchy(dim, k, levels, cells)
    g, n = h.finest, h.n_dofs()
    J = h.copy_jacobian(g).tocsr()
    A = J.T.tocsr() if transpose else J
    block = n // (k + 1)
    R = (block - (dim + 1) * h.sizes(g)["n_cells"]) // dim
    nodes = rng.choice(R, 40, replace=False)
    rows = np.array([a * block + l * R + i for i in nodes for a in range(k + 1) for l in range(dim)])
    for name, x in _vectors(rng, n).items():
        xt, b = torch.from_numpy(x).cuda(), torch.from_numpy(rng.standard_normal(n)).cuda()
        y, t = torch.full_like(xt, 7.0), torch.full_like(xt, 7.0)
        h.spmv(g, xt, y, transpose=transpose)
        h.defect(g, b, xt, t, transpose=transpose)
        y, t, b = y.cpu().numpy(), t.cpu().numpy(), b.cpu().numpy()
        ref = np.array([np.sum(A.data[A.indptr[r]:A.indptr[r + 1]].astype(np.longdouble)
                               * x[A.indices[A.indptr[r]:A.indptr[r + 1]]]) for r in rows])
        bound = _bound(A, x, rows, block, dim * R, dim) + 2.0**-51 * np.abs(ref).astype(float) + 2.0**-1060
        assert (np.abs(y[rows] - ref) <= bound).all(), name
        assert (np.abs(t[rows] - (b[rows] - ref)) <= bound + 2.0**-52 * np.abs(b[rows])).all(), name
    h.close()


@pytest.mark.parametrize("dim,k,levels,cells", [CASES[1], CASES[4]])
def test_nonfinite_entries(dim, k, levels, cells):
    import torch
    h, rng = _hierarchy(dim, k, levels, cells)
    g, n = h.finest, h.n_dofs()
    J = h.copy_jacobian(g).tocsr()
    x = rng.standard_normal(n)
    x[n // 3], x[n // 2] = np.nan, np.inf
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    h.spmv(g, torch.from_numpy(x).cuda(), y)
    y = y.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = J @ x
    assert np.array_equal(np.isnan(y), np.isnan(ref)) and np.array_equal(np.isinf(y), np.isinf(ref))
    fin = np.isfinite(ref)
    # FP64 sums of at most m terms on either side
    m = np.diff(J.indptr).max()
    bound = 2 * m * 2.0**-52 * (abs(J) @ np.where(np.isfinite(x), np.abs(x), 0.0))
    assert (np.abs(y - ref)[fin] <= bound[fin]).all()
    h.close()
