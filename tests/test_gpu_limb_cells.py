"""Cell solves over FP64 inverses kept as two-limb integers: one sweep from zero against the 32-column sweep, which
multiplies the FP64 inverses in FP64, for cells of one to three row pairs per lane, few and many cells (eight warps
to one per cell), both directions, and right-hand sides over many magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 1, 2, (3, 2)), (2, 1, 5, (16, 4)), (2, 2, 2, (5, 3)), (2, 2, 4, (10, 4)), (3, 0, 2, (3, 2, 2)),
         (3, 0, 2, (16, 4, 4)), (3, 1, 2, (2, 3, 2)), (3, 1, 2, (7, 4, 3))]


def _columns(rng, n):
    d = rng.standard_normal((32, n))
    for o in (0, 16):
        d[o + 1] *= np.exp2(rng.integers(-60, 60, n))
        d[o + 2] *= np.exp2(-200.0 * np.arange(n) / n)
        d[o + 3] *= rng.random(n) < 0.02
        d[o + 4] *= 2.0**-990   # below what the integers hold
        d[o + 5] = 0.0
        d[o + 6] *= 2.0**900
    return d


@pytest.mark.parametrize("dim,k,levels,cells", CASES)
def test_sweep_from_zero(dim, k, levels, cells):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, levels, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), inv_precision="f64"))
    rng = np.random.default_rng(8)
    h.assemble_jacobian(torch.from_numpy(0.3 * rng.standard_normal(h.n_dofs())).cuda())
    h.factor_cells()
    g, n = h.finest, h.n_dofs()
    R = _columns(rng, n)
    Rg = torch.from_numpy(R).cuda()
    f, a = torch.zeros_like(Rg[:16]), torch.zeros_like(Rg[16:])
    h.vanka_sweep_fused(g, Rg[:16].contiguous(), f, Rg[16:].contiguous(), a)
    fused = torch.cat([f, a]).cpu().numpy()
    # FP64 chains of m terms on either side: 2 m eps sum |J_T^{-1}| |t|; the integers: less than 2^-55 per term of the
    # largest row scale (pressure columns at the common offset of their cell) times the largest entry
    inv = np.abs(h.copy_cell_inverses(g))
    m = inv.shape[1]
    nt = m // (k + 1)
    vel = np.arange(m) % nt < dim * 3**dim
    v, p = inv[:, :, vel].max(2), inv[:, :, ~vel].max(2)
    scale = (v.max(1) * np.maximum(1.0, 4 * (p / v).max(1))).max()
    amp = max(inv.sum(1).max(), inv.sum(2).max())
    for c in list(range(7)) + list(range(16, 23)):
        d = torch.zeros_like(Rg[c])
        h.vanka_sweep(g, Rg[c].contiguous(), d, transpose=c >= 16)
        bound = (2 * m * 2.0**-52 * amp + m * 2.0**-55 * 4 * scale) * np.abs(R[c]).max() + 2.0**-1060
        assert np.abs(d.cpu().numpy() - fused[c]).max() <= bound, c
    h.close()
