"""FP32 Laplacian of large grids: extents that are no multiple of the tile, every copy width (n1 a
multiple of 4, even, odd; a field not aligned to the wider ones), blocks whose planes span two
tiles, each order.

Tolerance, from the arithmetic: a point's value is a sum of 6N + 1 <= 37 products in FP32, its
weights rounded to FP32 too: at most 40 2^-24 of sum |w| |f|, and |w_0| + 2 sum |w_p| <= 6.6 / h^2
per axis for every order.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,half_order,shift", [((95, 130, 131), 6, 0), ((95, 130, 131), 1, 0), ((130, 97, 250), 6, 0),
                                                ((130, 97, 250), 3, 0), ((132, 64, 301), 6, 0), ((132, 64, 301), 3, 1),
                                                ((64, 32, 913), 6, 2), ((129, 65, 160), 3, 0), ((200, 256, 57), 1, 0)])
def test_large_laplacian(n, half_order, shift):
    L = (0.21 * n[0], 0.25 * n[1], 0.3 * n[2])
    h = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        rng = np.random.default_rng(5)
        f = rng.standard_normal(n[::-1]).astype(np.float32)
        buf = torch.zeros(f.size + 4, dtype=torch.float32, device="cuda")
        x = buf[shift:shift + f.size].view(f.shape)
        x.copy_(torch.from_numpy(f))
        y = torch.full_like(x, float("nan"))
        B.of_laplacian_apply(h, B.OF_F32, x, y)
        x64, ref = x.double().contiguous(), torch.empty(f.shape, dtype=torch.float64, device="cuda")
        B.of_laplacian_apply(h, B.OF_F64, x64, ref)
        bound = 40 * 2.0 ** -24 * 6.6 * sum((m / l) ** 2 for m, l in zip(n, L)) * np.abs(f).max()
        assert float((y.double() - ref).abs().max()) <= bound
        # the FP64 sweep itself against the oracle, in one plane
        lap = O.laplacian(f.astype(np.float64), O.Grid(n, L, half_order))
        assert np.abs(ref.cpu().numpy()[3] - lap[3]).max() <= 1e-12 * np.abs(lap).max()
    finally:
        B.of_grid_destroy(h)
