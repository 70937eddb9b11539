"""Grid points 1e-9 inside or outside the cutoff sphere of an ion, which single precision cannot tell: the
self energy counts the same points as the nuclear charge does.

48 points lie at r^2 = 57 h^2 of an ion on a grid point.  With rc = 7.54 sigma they are 3e-13 of the sum;
the sums themselves (32 quadrature nodes of positive terms; the oracle's 10^4 terms) round to a few 1e-15:
tolerance 2e-14.  A point's own charge there is 5e-13 of the peak: tolerance 1e-13, as elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1.0, 1.1, 0.7])
@pytest.mark.parametrize("beyond", [1e-9, -1e-9])
def test_the_self_energy_counts_the_points_of_the_charge(step, beyond):
    n = (20, 18, 24)
    L = tuple(step * k for k in n)
    rc = step * np.sqrt(57.0 * (1.0 + beyond))
    sigma = rc / 7.54
    R, Z = np.array([[step * 9, step * 4, step * 11]]), np.array([3.0])
    h = B.of_grid_create(n, L, 6, torch.cuda.current_stream())
    try:
        grid = O.Grid(n, L, 6)
        b = torch.empty(grid.shape, dtype=torch.float64, device="cuda")
        e = B.of_pseudocharge(h, B.make_system(R, Z, sigma, rc), b)
        ref = O.pseudocharge(R, Z, sigma, rc, grid)
        assert np.max(np.abs(b.cpu().numpy() - ref)) <= 1e-13 * np.max(np.abs(ref))
        eref = O.self_energy(R, Z, sigma, rc, grid)
        assert abs(e - eref) <= 2e-14 * abs(eref)
    finally:
        B.of_grid_destroy(h)
