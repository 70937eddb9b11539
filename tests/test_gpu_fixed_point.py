"""The FP64 Laplacian's fixed-point sweep and its FP64 fallback against the oracle.

Bound, derived before the first run: a value keeps at least 53 bits relative to the largest of the
stretch of values around it (at most eight points away), so an output's error is at most
2^-53 sum|w| times the largest value within eight points, plus the FP64 rounding of the fallback's 37
operations and of the oracle's own sum: 80 * 2^-53 * sum|w| * local maximum covers all three."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
SIZES = [(5, 6, 7), (33, 17, 40), (32, 8, 8), (34, 9, 9), (70, 45, 3), (1, 1, 16), (96, 40, 24)]


def _local_max(a, r=8):
    m = np.abs(a)
    for ax in range(3):
        m = np.max([np.roll(m, s, ax) for s in range(-r, r + 1)], axis=0)
    return m


def _field(kind, shape, seed):
    x = W.random_field(shape, seed=seed)
    z, y, xx = np.meshgrid(*[np.arange(k) for k in shape], indexing="ij")
    if kind == "smooth":
        return W.random_field(shape, seed=seed, kind="smooth")
    if kind == "decay":                       # 1e-30 of range across the grid
        return x * 10.0 ** (-30.0 * (xx + y + z) / sum(shape))
    if kind == "spikes":                      # zeros, and values far above the rest
        x = np.where(x > 0.9, x * 1e12, 0.0)
        x[0, 0, 0] = 1e150
        return x
    return x * {"white": 1.0, "huge": 1e290, "tiny": 1e-300}[kind]


@pytest.mark.parametrize("kind", ["white", "smooth", "decay", "spikes", "huge", "tiny"])
@pytest.mark.parametrize("n", SIZES, ids=str)
def test_fp64_laplacian_is_accurate_at_every_point(n, kind):
    if not torch.cuda.is_available():
        pytest.fail("GPU test needs a CUDA device")
    for N, stretch in ((1, 1.0), (3, 1.1), (6, 1.0)):
        L = (0.2375 * n[0], 0.2375 * n[1] * stretch, 0.2375 * n[2])     # equal and unequal spacings
        h = B.of_grid_create(n, L, N, torch.cuda.current_stream())
        try:
            g = O.Grid(n, L, N)
            x = _field(kind, g.shape, seed=sum(n) + N)
            wsum = sum(2 * np.abs(O.fd_laplacian_weights(N, hd)).sum() for hd in g.h)
            ref = O.laplacian(x, g)
            bound = 80 * 2.0 ** -53 * wsum * _local_max(x) + 1e-322
            for offset in (0, 1):             # 16- and 8-byte aligned fields
                buf = torch.zeros(x.size + 2, dtype=torch.float64, device="cuda")
                xd = buf[offset:offset + x.size].view(x.shape)
                xd.copy_(torch.from_numpy(x))
                yd = torch.full_like(xd, float("nan"))
                B.of_laplacian_apply(h, B.OF_F64, xd, yd)
                assert np.all(np.abs(yd.cpu().numpy() - ref) <= bound), (N, offset)
        finally:
            B.of_grid_destroy(h)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_values_stay_local(bad):
    n = (40, 24, 24)
    h = B.of_grid_create(n, tuple(0.2375 * k for k in n), 6, torch.cuda.current_stream())
    try:
        x = torch.from_numpy(W.random_field((24, 24, 40), seed=1)).cuda()
        y0, y1 = torch.empty_like(x), torch.empty_like(x)
        B.of_laplacian_apply(h, B.OF_F64, x, y0)
        x[3, 4, 5] = bad
        B.of_laplacian_apply(h, B.OF_F64, x, y1)
        hit = ~torch.isfinite(y1)
        assert int(hit.sum()) == 37 and hit[3, 4, 5] and hit[3, 4, 11] and hit[21, 4, 5] and hit[3, 22, 5]
        assert torch.allclose(y0[~hit], y1[~hit], rtol=0, atol=1e-11)
    finally:
        B.of_grid_destroy(h)
