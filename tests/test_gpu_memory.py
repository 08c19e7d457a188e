"""Little device memory: copies that only save time are not made where they would not fit, are given back when a required
allocation fails, and the results stay within rounding."""
import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MESH = (3, 1, 2, (16, 4, 4), (2.5, 0.41, 0.41))


def _hierarchy(inv, X=None):
    import torch
    from paper_2107_10561_gb300 import Hierarchy, make_params
    h = Hierarchy(make_params(*MESH, inv_precision=inv))
    if X is None:
        X = torch.from_numpy(0.1 * np.random.default_rng(3).standard_normal(h.n_dofs())).cuda()
    h.assemble_jacobian(X)
    h.factor_cells()
    return h, X


@contextlib.contextmanager
def _only(left):
    """Takes all device memory but `left` bytes."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(max(0, torch.cuda.mem_get_info()[0] - left), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        torch.cuda.synchronize()
        del hold
        torch.cuda.empty_cache()


def _rows(a, b):
    return float((a - b).abs().max() / b.abs().max())


def test_cell_solves_without_room_and_given_back():
    import torch
    rng = np.random.default_rng(5)
    h, X = _hierarchy("f64")
    h2, _ = _hierarchy("f64", X)
    n, g = h.n_dofs(), h.finest
    r = torch.from_numpy(rng.standard_normal(n)).cuda()
    fast, slow, after, x, y = (torch.zeros_like(r) for _ in range(5))
    h.vanka_sweep(g, r, fast)  # makes the copy: 2,048 cells of 170 x 170, 473 MB
    with _only(256 << 20):
        h2.vanka_sweep(g, r, slow)  # no room for one
    assert _rows(slow, fast) < 1e-12
    h2.close()
    # a Krylov basis of 61 vectors (63 MB) into 40 MB: the copy goes
    with _only(40 << 20):
        assert h.gmres_solve(r, x, rtol=1e-9)["converged"]
        h.vanka_sweep(g, r, after)
    assert _rows(after, fast) < 1e-12
    h.spmv(g, x, y)
    assert float((y - r).norm() / r.norm()) < 2e-9
    h.close()


def test_multi_products_without_room():
    import torch
    h, X = _hierarchy("bf16")
    B = torch.from_numpy(np.random.default_rng(6).standard_normal((32, h.n_dofs()))).cuda()
    fast, slow = torch.zeros_like(B), torch.zeros_like(B)
    h.gmres_solve_multi(B, fast, rtol=1e-9, restart=8, max_iter=60)
    h.close()
    # room for the vectors (0.95 GB) but not for the operands of the products (0.41 GB) as well
    h, _ = _hierarchy("bf16", X)
    with _only(1200 << 20):
        h.gmres_solve_multi(B, slow, rtol=1e-9, restart=8, max_iter=60)
    assert _rows(slow, fast) < 1e-7
    h.close()
