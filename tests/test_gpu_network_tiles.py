"""Convolution layers of the learned preconditioner at the edges of their tiles: x-rows that are
no multiple of the 8 points of a group, fewer groups than a tile, more blocks than rows of tiles
and fewer, axes shorter than the 3 x 3 x 3 taps' own width.

Tolerances: as for the network and its gradients on the larger grids, four to five times the
error of an FP64 oracle whose input and activations are rounded to BF16 (0.37 % RMS in the output,
<= 0.1 % in each weight gradient).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import precond as NP  # noqa: E402
from paper_1412_8250_gb300 import binding as B  # noqa: E402
from test_gpu_precond import GROUPS, _field, _flat, _params, _unflat  # noqa: E402
import oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu
H = 0.2375


def _grid(n, half_order):
    L = tuple(H * m for m in n)
    return B.of_grid_create(n, L, half_order, torch.cuda.current_stream()), O.Grid(n, L, half_order)


@pytest.mark.parametrize("n", [(8, 16, 16), (17, 12, 31), (130, 14, 13), (13, 150, 14), (121, 16, 15)])
def test_forward_on_ragged_tiles(n):
    h, grid = _grid(n, 1)
    P = _params(3)
    net = B.of_precond_create(_flat(P))
    try:
        r = _field(grid.shape, 7)
        z = torch.empty(grid.shape, dtype=torch.float32, device="cuda")
        B.of_precond_apply(h, net, torch.tensor(r, dtype=torch.float32, device="cuda"), z)
        ref = NP.apply(P, r)
        err = z.cpu().numpy().astype(np.float64) - ref
        assert np.sqrt(np.mean(err ** 2)) <= 1.5e-2 * np.sqrt(np.mean(ref ** 2))
        assert np.abs(err).max() <= 2e-2 * np.abs(ref).max()
    finally:
        B.of_precond_destroy(net)
        B.of_grid_destroy(h)


def test_gradients_on_ragged_tiles():
    h, grid = _grid((33, 20, 17), 6)
    P = _params(5)
    net = B.of_precond_create(_flat(P))
    try:
        r = _field(grid.shape, 11)
        loss, g = B.of_precond_loss_grad(h, net, torch.tensor(r, dtype=torch.float32, device="cuda"))
    finally:
        B.of_precond_destroy(net)
        B.of_grid_destroy(h)
    ref_loss, ref = NP.loss_and_grads(P, r, grid)
    assert abs(loss - ref_loss) <= 1e-3 * abs(ref_loss)
    G = _unflat(g, P)
    total = np.sqrt(sum(np.sum(ref[k] ** 2) for k in GROUPS))
    for k in GROUPS:
        bar = 5e-3 * (total if k == "b3" else np.linalg.norm(ref[k]))
        assert np.linalg.norm(G[k] - ref[k]) <= bar, k
