"""The 32-column product with J on the tensor cores: R - J D as the additive sweep uses it, for every number
of velocity rows per node, meshes with full and ragged neighbour lists, and D over magnitudes that cross
digits from node to node. With R = J D from the FP64 CSR product a sweep changes D by rounding only,
amplified by the cell inverses."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 0, (3, 2)), (2, 1, (4, 3)), (2, 2, (5, 3)), (3, 0, (3, 2, 2)), (3, 1, (2, 3, 2))]


def _hierarchy(dim, k, cells):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, 2, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), inv_precision="f64"))
    rng = np.random.default_rng(3)
    h.assemble_jacobian(torch.from_numpy(0.3 * rng.standard_normal(h.n_dofs())).cuda())
    h.factor_cells()
    return h, rng


def _spread(kind, rng, n):
    d = rng.standard_normal((32, n))
    if kind == "columns":  # every column at its own magnitude, some zero
        d *= 10.0 ** rng.integers(-200, 200, (32, 1))
        d[5] = 0.0
    if kind == "decay":    # falls off along the numbering, so neighbours differ by digits
        d *= 2.0 ** (-60.0 * np.arange(n) / n)
    if kind == "sparse":
        d *= rng.random((32, n)) < 0.03
    return d


@pytest.mark.parametrize("dim,k,cells", CASES)
@pytest.mark.parametrize("kind", ["normal", "columns", "decay", "sparse"])
@pytest.mark.parametrize("fused", [False, True])
def test_product_against_csr(dim, k, cells, kind, fused):
    import torch
    h, rng = _hierarchy(dim, k, cells)
    n, g = h.n_dofs(), h.finest
    J = h.copy_jacobian(g)
    D = _spread(kind, rng, n)
    JD = np.stack([(J.T if fused and c >= 16 else J) @ D[c] for c in range(32)])
    # R = J D in FP64: what is left of R - J D is rounding, and the sweep returns J_T^{-1} of it
    R, Dg = torch.from_numpy(JD).cuda(), torch.from_numpy(D).cuda()
    if fused:
        f, a = Dg[:16].clone(), Dg[16:].clone()
        h.vanka_sweep_fused(g, R[:16].contiguous(), f, R[16:].contiguous(), a)
        out = torch.cat([f, a]).cpu().numpy()
    else:
        out = Dg.clone()
        h.vanka_sweep_multi(g, R, out)
        out = out.cpu().numpy()
    inv = h.copy_cell_inverses(g)
    # |R - J D| <= 2 gamma_m |J||D| per row for an FMA chain of m <= 1000 terms on either side (gamma_m = m eps);
    # a cell inverse and the weights (sum to one) turn that into at most the largest row sum of |J_T^{-1}|
    eps, rows = 2.0**-52, np.diff(J.indptr).max()
    A = abs(J)
    for c in range(32):
        bound = 2 * rows * eps * ((A.T if fused and c >= 16 else A) @ abs(D[c])).max()
        amp = abs(inv).sum(1 if fused and c >= 16 else 2).max()
        assert np.abs(out[c] - D[c]).max() <= bound * amp, c
    h.close()


def test_nonfinite_columns_stay_in_their_rows():
    import torch
    h, rng = _hierarchy(2, 2, (5, 3))
    n, g = h.n_dofs(), h.finest
    D = rng.standard_normal((32, n))
    D[3, n // 2], D[20, n // 3] = np.nan, np.inf
    R = torch.from_numpy(rng.standard_normal((32, n))).cuda()
    multi = torch.from_numpy(D).cuda()
    h.vanka_sweep_multi(g, R, multi)
    for c in (3, 4, 20):
        one = torch.from_numpy(D[c].copy()).cuda()
        h.vanka_sweep(g, R[c].contiguous(), one)
        assert torch.equal(torch.isfinite(multi[c]), torch.isfinite(one)), c
    h.close()
