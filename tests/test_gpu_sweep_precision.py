"""The FP64 Laplacian is as accurate at each point as the values of that point's own stencil allow, whatever
stands elsewhere in the brick that the sweep shares an exponent over: compact support next to large
values, fields that fall by powers of ten per point, subnormal values.

Bound: the oracle's sum of 6N + 1 <= 37 products rounds to at most 40 2^-53 of S = sum |w| |f| over the
point's stencil.  In fixed point (unit d, the largest of a point's own and next values >= 2^53 d) the
sum is cut off by at most 5.7 d / h^2 per conversion, of which unequal spacings have three, and the
values by at most d each, 21.1 d / h^2 over all weights: 38.2 d / h^2 against 2^-53 S >= 1.5 d / h^2, or
26 2^-53 S; with the four roundings of the scale and the unequal spacings' 1.1^2 below 36 2^-53 S.
40 2^-53 S for each of the two; results below the normal range round to 2^-1075 per product.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _halo(shape):
    # one plane holds 1e30 and, more than eight points away along x, 1.0; the rest is zero
    f = np.zeros(shape)
    f[8, 4, 3], f[8, 4, min(24, shape[2] - 1)] = 1e30, 1.0
    return f


def _fields(shape, seed):
    r = W.random_field(shape, seed=seed)
    z, y, x = np.meshgrid(*[np.arange(k) for k in shape], indexing="ij")
    yield "halo", _halo(shape)
    yield "tenfold", 10.0 ** -(x % 16 + z % 5) * (1.0 + 0.5 * r)
    yield "half", np.where(x < shape[2] // 2, r, 0.0)
    yield "spike", 1e-9 * r + (x + y + z == 5) * 1.0
    yield "nodes", np.sin(2 * np.pi * x / shape[2]) * np.cos(2 * np.pi * z / shape[0]) + 1e-12 * r
    yield "subnormal", 1e-310 * r
    yield "tiny beside", np.where(z < 3, r, 1e-320 * r)


@pytest.mark.parametrize("n", [(40, 24, 32), (33, 17, 20), (32, 9, 9), (96, 40, 56), (200, 88, 64)], ids=str)
@pytest.mark.parametrize("half_order", [1, 3, 6])
@pytest.mark.parametrize("stretch", [1.0, 1.1])
def test_laplacian_is_accurate_to_its_stencil(n, half_order, stretch):
    L = (0.2375 * n[0], 0.2375 * n[1] * stretch, 0.2375 * n[2])
    h = B.of_grid_create(n, L, half_order, torch.cuda.current_stream())
    try:
        g = O.Grid(n, L, half_order)
        for name, f in _fields(g.shape, sum(n) + half_order):
            S = np.zeros(g.shape)
            for a in range(3):
                w = np.abs(O.fd_laplacian_weights(half_order, g.h[a]))
                S += w[0] * np.abs(f)
                for p in range(1, half_order + 1):
                    S += w[p] * (np.roll(np.abs(f), p, 2 - a) + np.roll(np.abs(f), -p, 2 - a))
            xd = torch.from_numpy(f).cuda()
            yd = torch.full_like(xd, float("nan"))
            B.of_laplacian_apply(h, B.OF_F64, xd, yd)
            err = np.abs(yd.cpu().numpy() - O.laplacian(f, g))
            assert np.all(err <= 80 * 2.0 ** -53 * S + 80 * 2.0 ** -1074), (name, np.max(err / (S + 1e-320)))
    finally:
        B.of_grid_destroy(h)
