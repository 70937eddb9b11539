"""FP32 Laplacian of large grids with a one-point last column and row of tiles; every case is one that the
tile-walking kernel takes (tiles of 64 x 32 points, at least 6 planes per SM, more than half of the
tiles' points on the grid).  Tolerance: as for the other large FP32 sweeps, 40 2^-24 sum |w| |f|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,half_order", [((193, 129, 160), 3), ((193, 129, 131), 6), ((193, 65, 160), 1), ((321, 97, 101), 6)])
def test_large_laplacian_with_one_point_tiles(n, half_order):
    tiles = -(-n[0] // 64) * -(-n[1] // 32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert tiles * n[2] >= 6 * sms and 2 * n[0] * n[1] > tiles * 64 * 32 and n[0] % 64 == 1 and n[1] % 32 == 1
    L = (0.21 * n[0], 0.25 * n[1], 0.3 * n[2])
    h = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        f = np.random.default_rng(5).standard_normal(n[::-1]).astype(np.float32)
        x = torch.from_numpy(f).cuda()
        y = torch.full_like(x, float("nan"))
        B.of_laplacian_apply(h, B.OF_F32, x, y)
        lap = O.laplacian(f.astype(np.float64), O.Grid(n, L, half_order))
        bound = 40 * 2.0 ** -24 * 6.6 * sum((m / l) ** 2 for m, l in zip(n, L)) * np.abs(f).max()
        assert np.abs(y.cpu().numpy() - lap).max() <= bound
    finally:
        B.of_grid_destroy(h)
