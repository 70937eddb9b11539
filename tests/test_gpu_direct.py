"""The direct (Fourier-diagonalised) corrections of the mixed-precision solves against the oracle's
exact discrete solution, at the extents where the transforms differ: one point, small and large
primes, every unrolled radix, odd row counts (rows are transformed in pairs), long lines with fewer
lines per tile, and an axis beyond the transforms' limit, which keeps the multigrid solver.

Tolerances: a solve to a true relative residual of 1e-12 agrees with the exact solution to 1e-9 of its
largest value, the bar of the other solves (the longest wave of these grids amplifies the residual by
less than 1e3 relative to the solution)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
H = 0.2375
SIZES = [(1, 1, 16), (2, 3, 5), (7, 9, 10), (11, 13, 17), (31, 37, 41), (45, 50, 54), (33, 1, 12),
         (12, 16, 49), (96, 40, 20), (131, 8, 6), (6, 4, 600), (4, 1200, 3)]


def _opts(tol):
    o = B.of_default_solve_opts()
    o.tol, o.precision = tol, B.OF_F32
    return o


def _grid(n, N):
    if not torch.cuda.is_available():
        pytest.fail("GPU test needs a CUDA device")
    L = tuple(H * k for k in n)
    return B.of_grid_create(n, L, N, torch.cuda.current_stream()), O.Grid(n, L, N)


@pytest.mark.parametrize("n", SIZES, ids=str)
@pytest.mark.parametrize("N", [1, 6])
def test_direct_poisson_and_shifted_solves(n, N):
    h, g = _grid(n, N)
    try:
        rho = W.random_field(g.shape, seed=3) + W.random_field(g.shape, seed=5, kind="smooth")
        ref = O.poisson_solve(rho, g)
        phi = torch.from_numpy(W.random_field(g.shape, seed=4)).cuda()       # a guess that is not zero
        info = B.of_poisson_solve(h, torch.from_numpy(rho).cuda(), phi, _opts(1e-12))
        assert info.rel_residual <= 1e-12 and info.iterations <= 6
        assert np.abs(phi.cpu().numpy() - ref).max() <= 1e-9 * np.abs(ref).max()
        for Q in (-0.470923 - 0.465392j, -0.511699 - 0.0266195j, 0.066051 - 0.259678j):
            P, kf2 = 0.108403 + 0.079657j, 2.5
            ref = O.kernel_solve(rho, g, kf2, P, Q)
            Wc = torch.zeros(g.shape + (2,), dtype=torch.float64, device="cuda")
            info = B.of_kernel_solve(h, torch.from_numpy(rho).cuda(), [P], [Q], kf2, Wc, _opts(1e-12))
            w = Wc.cpu().numpy()
            assert info.rel_residual <= 1e-12
            assert np.abs(w[..., 0] + 1j * w[..., 1] - ref).max() <= 1e-9 * np.abs(ref).max()
    finally:
        B.of_grid_destroy(h)


def test_an_axis_beyond_the_transforms_keeps_the_multigrid_solver():
    h, g = _grid((2304, 16, 16), 6)
    try:
        rho = W.random_field(g.shape, seed=3) + W.random_field(g.shape, seed=5, kind="smooth")
        phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        info = B.of_poisson_solve(h, torch.from_numpy(rho).cuda(), phi, _opts(1e-10))
        assert info.rel_residual <= 1e-10 and info.iterations > 6
    finally:
        B.of_grid_destroy(h)


def test_a_singular_mode_is_left_to_the_krylov_solver():
    # Q = -a l(k) for one mode k: the symbol vanishes there, so a right-hand side without that mode is
    # solvable and one made of it is not; neither may return non-finite values
    n, N, kf2 = (8, 8, 8), 1, 1.0
    h = B.of_grid_create(n, (8.0, 8.0, 8.0), N, torch.cuda.current_stream())
    try:
        g = O.Grid(n, (8.0, 8.0, 8.0), N)
        lam = float(-O.laplacian_symbol(g)[0, 0, 4])       # 4: exact in binary
        x = np.arange(8)
        f = np.cos(np.pi * x)[None, None, :] * np.ones((8, 8, 1))
        Wc = torch.zeros((8, 8, 8, 2), dtype=torch.float64, device="cuda")
        o = _opts(1e-10)
        o.max_iter = 50
        st = None
        try:
            B.of_kernel_solve(h, torch.from_numpy(f.copy()).cuda(), [1.0 + 0j], [-lam + 0j], kf2, Wc, o)
        except B.OfError as e:
            st = e.status
        assert st in (B.OF_EBREAKDOWN, B.OF_ENOCONV)
        assert torch.isfinite(Wc).all()
    finally:
        B.of_grid_destroy(h)
