"""FP64 CG in one launch: grids of one brick and of many, extents that are no multiple of a brick's,
rows of odd length, equal and unequal spacings, each order, against the exact discrete solution;
the residual it reports against the definition.

Tolerance: the error of a solve to relative residual t is at most cond(A) t; with spacings within a
factor of 1.5 and at most 50 points per axis cond(A) <= 4 n^2 <= 10^4, and t = 1e-13.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,half_order", [((13, 13, 13), (0.25, 0.25, 0.25), 6), ((31, 9, 7), (0.2, 0.25, 0.3), 3),
                                            ((33, 17, 50), (0.25, 0.25, 0.25), 6), ((45, 50, 18), (0.25, 0.2, 0.3), 6),
                                            ((32, 24, 16), (0.25, 0.25, 0.25), 3), ((47, 41, 5), (0.25, 0.25, 0.25), 1),
                                            ((50, 49, 48), (0.3, 0.25, 0.2), 1)])
def test_poisson(n, h, half_order):
    L = tuple(a * m for a, m in zip(h, n))
    g = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        grid = O.Grid(n, L, half_order)
        rho = W.random_field(grid.shape, seed=3)
        phi = torch.from_numpy(W.random_field(grid.shape, seed=4)).cuda()   # a guess that is not zero
        o = B.of_default_solve_opts()
        o.tol = 1e-13
        info = B.of_poisson_solve(g, torch.from_numpy(rho).cuda(), phi, o)
        ref = O.poisson_solve(rho, grid)
        got = phi.cpu().numpy()
        assert info.rel_residual <= 1e-13
        assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()
        b = 4 * np.pi * (rho - rho.mean())
        # the reported residual is the true one, up to the rounding of the oracle's Laplacian
        assert np.linalg.norm(b + O.laplacian(got, grid)) <= 1e-12 * np.linalg.norm(b)
        # a cell repeated with a lower iteration limit stops there
        phi2 = torch.zeros_like(phi)
        o.max_iter = 2
        info = B.of_poisson_solve(g, torch.from_numpy(rho).cuda(), phi2, o, allow=(B.OF_ENOCONV,))
        assert info.iterations == 2 and info.rel_residual > 1e-13
    finally:
        B.of_grid_destroy(g)
