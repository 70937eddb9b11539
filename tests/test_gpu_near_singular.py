"""Shifted systems whose symbol a l(k) + Q nearly vanishes at one mode: a correction in FP32, which knows
that mode's symbol to a few 2^-24 of a l alone, must not make the caller's guess worse.  The shifts
are real and negative, 1e-8 from one mode's eigenvalue relative to it, where FP32 arithmetic (its
products exact) sees 6e-12 .. 3e-11.

At most three iterations: the direct passes alone (COCG, which continues after them, does not lower
the residual in every iteration).  The residual after the solve, by the oracle, is at most the guess's, and the one that the solve reports:
both up to 1e-6 of the right-hand side, the rounding of a field whose singular part may be 1e8 times
the rest (2^-53 of sum |w| |x| <= 2e9).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
N3, H = (12, 10, 14), 0.2375


@pytest.mark.parametrize("kf2,q", [(2.25, 113.67670440673828), (1.5, 170.51506042480469), (2.45, 56.77835464477539)])
@pytest.mark.parametrize("max_iter", [1, 2, 3])
def test_a_nearly_singular_mode_does_not_spoil_the_guess(kf2, q, max_iter):
    L = tuple(H * k for k in N3)
    h = B.of_grid_create(N3, L, 6, torch.cuda.current_stream())
    try:
        g = O.Grid(N3, L, 6)
        f = W.random_field(g.shape, seed=1)
        guess = np.stack([W.random_field(g.shape, seed=2), W.random_field(g.shape, seed=3)], -1) * 1e-3
        P, Q = 1.0 + 0.5j, -q + 0.0j

        def residual(w):
            c = w[..., 0] + 1j * w[..., 1]
            lap = O.laplacian(c.real, g) + 1j * O.laplacian(c.imag, g)
            return np.linalg.norm(P * f + lap / kf2 - Q * c) / np.linalg.norm(P * f)

        Wc = torch.from_numpy(guess).cuda()
        o = B.of_default_solve_opts()
        o.tol, o.precision, o.max_iter = 1e-12, B.OF_F32, max_iter
        info = B.of_kernel_solve(h, torch.from_numpy(f).cuda(), [P], [Q], kf2, Wc, o,
                                 allow=(B.OF_ENOCONV, B.OF_EBREAKDOWN))
        after = residual(Wc.cpu().numpy())
        assert after <= residual(guess) + 1e-6
        assert abs(info.rel_residual - after) <= 1e-6
    finally:
        B.of_grid_destroy(h)
