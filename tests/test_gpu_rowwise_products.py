"""J x row by row: the error of every entry against the sum of |J| |x| in its own row, for x whose velocity
components, time nodes and pressures differ by orders of magnitude, for x that is large at single entries, and for
linearisations at rest, in a channel flow and in a perturbed one (blocks of J that vanish, nearly vanish or do not)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 0, 3, (6, 3)), (2, 1, 3, (6, 3)), (3, 0, 2, (3, 2, 2)), (3, 1, 2, (4, 3, 2)), (3, 1, 3, (14, 4, 4)),
         (3, 2, 2, (3, 2, 2)), (2, 2, 5, (6, 3)), (2, 2, 5, (10, 4))]


def _classes(n, k, dim, R):
    """Velocity component or pressure (dim) and time node of every unknown."""
    block = n // (k + 1)
    v = np.arange(n) % block
    return np.minimum(v // R, dim), np.arange(n) // block


def vectors(rng, n, comp, time, dim):
    x = rng.standard_normal(n)
    out = {"normal": x}
    for s in (1e-2, 1e-5, 1e-8):
        out[f"cross flow {s}"] = x * np.where(comp == 0, 1.0, s)
        out[f"pressure {1 / s}"] = x * np.where(comp == dim, 1 / s, 1.0)
        out[f"velocity pressure {s}"] = x * np.where(comp == dim, s, 1.0)
        out[f"time {s}"] = x * s ** time
    out["decay"] = x * np.exp2(-60.0 * np.arange(n) / n)
    out["wide"] = x * np.exp2(rng.integers(-20, 20, n))
    out["sparse"] = np.where(rng.random(n) < 0.02, x, 0.0)
    out["spikes"] = x * np.where(rng.random(n) < 0.01, 1e12, 1.0)
    return out


def linearisation(h, kind, rng, k, dim, R):
    X = np.zeros(h.n_dofs())
    comp, _ = _classes(X.size, k, dim, R)
    if kind == "channel":  # streamwise only: the blocks between components vanish or nearly do
        node = (np.arange(X.size) % (X.size // (k + 1))) % R
        X = np.where(comp == 0, 0.3 * np.sin(np.pi * node / R), 0.0)
    if kind == "perturbed":
        X = np.where(comp < dim, 0.3 * rng.standard_normal(X.size), 0.0)
    return X


@pytest.mark.parametrize("dim,k,levels,cells", CASES)
@pytest.mark.parametrize("kind", ["rest", "channel", "perturbed"])
@pytest.mark.parametrize("tau", [1e-2, 1e-5])
def test_rows(dim, k, levels, cells, kind, tau):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(dim, k, levels, cells, (2.2, 0.41) if dim == 2 else (2.5, 0.41, 0.41), tau=tau))
    rng = np.random.default_rng(17)
    g, n = h.finest, h.n_dofs()
    R = (n // (k + 1) - (dim + 1) * h.sizes(g)["n_cells"]) // dim
    h.assemble_jacobian(torch.from_numpy(linearisation(h, kind, rng, k, dim, R)).cuda())
    J = h.copy_jacobian(g).tocsr()
    comp, time = _classes(n, k, dim, R)
    rows = rng.choice(n, 400, replace=False)
    for transpose in (False, True):
        A = (J.T.tocsr() if transpose else J)[rows]
        m = np.diff(A.indptr)
        for name, x in vectors(rng, n, comp, time, dim).items():
            xt = torch.from_numpy(x).cuda()
            y = torch.full_like(xt, 7.0)
            h.spmv(g, xt, y, transpose=transpose)
            p = A.data.astype(np.longdouble) * x[A.indices]
            at = np.concatenate([[0], np.cumsum(m)[:-1]])
            ref, S = np.add.reduceat(p, at), np.add.reduceat(np.abs(p), at)
            # what a chain of m FP64 multiply-adds is held to
            bound = (m + 4) * 2.0**-53 * S.astype(float) + 2.0**-1060
            err = np.abs(y.cpu().numpy()[rows] - ref)
            assert (err <= bound).all(), (name, transpose, float((err / bound).max()))
    h.close()
