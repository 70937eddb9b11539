"""FP64 Laplacian where L / n rounds to different spacings on the axes though L = H n: one scale for
all axes; and where the spacings differ for good.

Tolerance: the three scales 1 / h^2 differ by at most 2^-50 and their mean from each by half that;
weights, sum and scale round to 2^-53 a few times each and a staged value is within 2^-53 of its
stretch's largest: 8 2^-52 of sum |w| |f| <= 6.6 / h^2 per axis times the largest |f|, the oracle's own
sum of 37 products as much again.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu
H = 7.6 / 32


@pytest.mark.parametrize("n,stretch", [((48, 32, 20), 1.0), ((16, 96, 20), 1.0), ((41, 24, 50), 1.0), ((32, 16, 24), 1 + 1e-12)])
@pytest.mark.parametrize("half_order", [1, 3, 6])
def test_laplacian_with_rounded_spacings(n, stretch, half_order):
    L = (H * n[0], H * n[1], stretch * H * n[2])
    spacings = {l / m for l, m in zip(L, n)}
    assert len(spacings) > 1   # what the case is about
    h = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        f = np.random.default_rng(2).standard_normal(n[::-1])
        x = torch.from_numpy(f).cuda()
        y = torch.empty_like(x)
        B.of_laplacian_apply(h, B.OF_F64, x, y)
        ref = O.laplacian(f, O.Grid(n, L, half_order))
        bound = 16 * 2.0 ** -52 * 6.6 * sum((m / l) ** 2 for m, l in zip(n, L)) * np.abs(f).max()
        assert np.abs(y.cpu().numpy() - ref).max() <= bound
    finally:
        B.of_grid_destroy(h)
