"""FP64 CG in one cooperative launch: the path on which its blocks give up waiting, and the grids that take
bricks of eight planes (more than three two-plane bricks per SM), whose last brick is not full.

Tolerance: as for the smaller grids, 1e-9 of the largest value at a residual of 1e-13 (cond(A) <= 2 n^2
<= 10^4 with equal spacings and at most 66 points per axis)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _solve(g, rho, tol=1e-13):
    o = B.of_default_solve_opts()
    o.tol = tol
    phi = torch.zeros(rho.shape, dtype=torch.float64, device="cuda")
    info = B.of_poisson_solve(g, torch.from_numpy(rho).cuda(), phi, o)
    return phi.cpu().numpy(), info


@pytest.mark.parametrize("n", [(13, 12, 11), (64, 63, 62)], ids=str)
def test_a_wait_that_runs_out_gives_a_timeout_status(n):
    g = B.of_grid_create(n, tuple(0.25 * k for k in n), 6, torch.cuda.current_stream())
    try:
        rho = W.random_field(n[::-1], seed=3)
        ref, _ = _solve(g, rho)
        for _ in range(2):
            B.of_grid_set_wait_limit(g, 0.0)
            with pytest.raises(B.OfError) as e:
                _solve(g, rho)
            assert e.value.status == B.OF_ETIMEOUT, str(e.value)
            B.of_grid_set_wait_limit(g, 2.0)
            again, info = _solve(g, rho)
            assert np.array_equal(again, ref) and info.rel_residual <= 1e-13
        with pytest.raises(B.OfError):
            B.of_grid_set_wait_limit(g, -1.0)
    finally:
        B.of_grid_destroy(g)


@pytest.mark.parametrize("n", [(64, 64, 64), (63, 66, 61)], ids=str)
@pytest.mark.parametrize("half_order", [1, 3, 6])
def test_bricks_of_eight_planes(n, half_order):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    columns = -(-n[0] // 32) * -(-n[1] // 8)
    assert columns * -(-n[2] // 2) > 3 * sms and columns * -(-n[2] // 8) <= 2 * sms
    L = tuple(0.25 * k for k in n)
    g = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        rho = W.random_field(n[::-1], seed=5)
        before = B.of_launch_count()
        got, info = _solve(g, rho)
        assert B.of_launch_count() - before < 20      # one launch holds the iterations
        ref = O.poisson_solve(rho, O.Grid(n, L, half_order))
        assert info.iterations > 20 and np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()
    finally:
        B.of_grid_destroy(g)
