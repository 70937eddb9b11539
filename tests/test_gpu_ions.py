"""Ion terms where their kernels branch: cutoffs on both sides of the separable self terms' limits
(7.53 and 9.2 widths), cells smaller than the ions' boxes (every image), boxes whose extent is not a
multiple of the strips and tiles, an ion on a grid point.

Tolerances: those of the other ion tests -- charge 1e-13 of its peak, self energy 1e-12 relative, forces
1e-11 (sums of order 1e5 FP64 terms of either sign)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma,rc", [(0.9, 6.0), (0.9, 6.7), (0.9, 6.85), (0.9, 8.2), (0.9, 8.4), (0.5, 5.5)])
@pytest.mark.parametrize("n,L", [((20, 14, 26), (7.0, 5.0, 9.0)), ((9, 40, 33), (3.0, 12.0, 10.0))], ids=str)
def test_ion_terms(n, L, sigma, rc):
    if not torch.cuda.is_available():
        pytest.fail("GPU test needs a CUDA device")
    cell = W.small_cell(n=n, L=L, sigma=sigma, rc=rc, seed=5)
    cell.R[1] = [2 * L[0] / n[0], 3 * L[1] / n[1], 0.0]
    grid = O.Grid(n, L, 6)
    h = B.of_grid_create(n, L, 6, torch.cuda.current_stream())
    try:
        sysd = B.make_system(cell.R, cell.Z, sigma, rc)
        b = torch.empty(grid.shape, dtype=torch.float64, device="cuda")
        e = B.of_pseudocharge(h, sysd, b)
        ref = O.pseudocharge(cell.R, cell.Z, sigma, rc, grid)
        assert np.max(np.abs(b.cpu().numpy() - ref)) <= 1e-13 * np.max(np.abs(ref))
        eref = O.self_energy(cell.R, cell.Z, sigma, rc, grid)
        assert abs(e - eref) <= 1e-12 * abs(eref)
        phi = W.random_field(grid.shape, seed=9, kind="smooth") + 0.1 * W.random_field(grid.shape, seed=3)
        F = B.of_forces(h, sysd, None, torch.from_numpy(phi).cuda())
        Fref = O.forces(phi, cell.R, cell.Z, sigma, rc, grid)
        assert np.max(np.abs(F - Fref)) <= 1e-11 * max(1.0, np.max(np.abs(Fref)))
    finally:
        B.of_grid_destroy(h)
