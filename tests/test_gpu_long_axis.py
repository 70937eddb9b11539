"""The solvers that serve grids beyond the direct solves' 2048 points per axis: multigrid-preconditioned
CG and COCG, and the V-cycles of the preconditioned NLCG, with the profile showing that they ran.

Tolerances: 1e-9 of the largest value at a residual of 1e-12 (the longest wave of the data amplifies by
119, the longest of the cell by 63 times more).  Everything here is reproducible to the bit; the NLCG's energy and
gradient fall.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
from paper_1412_8250_gb300 import binding as B, functionals as Fn, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
N3 = (16, 16, 2304)
L3 = tuple(0.2375 * k for k in N3)


def _launched(h):
    return {s["kernel"]: s["launches"] for s in B.of_profile_read(h)}


def _rhs(g):
    # waves 8 to 40 along the long axis, and noise without its longest waves
    x = np.arange(N3[2]) * (2 * np.pi / N3[2])
    long = sum(np.cos(k * x + k) for k in (8, 13, 29, 40))[:, None, None]
    r = np.fft.rfft(W.random_field(g.shape, seed=3), axis=0)
    r[:8] = 0.0
    return np.fft.irfft(r, n=N3[2], axis=0) + long


def test_multigrid_solves_beyond_the_direct_ones():
    out = []
    for _ in range(2):
        h = B.of_grid_create(N3, L3, 6, torch.cuda.current_stream())
        try:
            g = O.Grid(N3, L3, 6)
            rho, o = _rhs(g), B.of_default_solve_opts()
            o.tol, o.precision = 1e-12, B.OF_F32
            B.of_profile_enable(h, 1)
            phi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
            B.of_poisson_solve(h, torch.from_numpy(rho).cuda(), phi, o)
            P, Q, kf2 = Fn.P00[0], Fn.Q00[0], 0.9
            Wc = torch.zeros(g.shape + (2,), dtype=torch.float64, device="cuda")
            B.of_kernel_solve(h, torch.from_numpy(rho).cuda(), [P], [Q], kf2, Wc, o)
            ran = _launched(h)
            assert ran.get("mg_smooth", 0) + ran.get("mg_pcg_pass_graph", 0) > 0, ran
            assert ran.get("mg_cocg_pass_graph", 0) > 0 and "fft_direct_solve" not in ran, ran
            out.append((phi.cpu().numpy(), Wc.cpu().numpy()))
        finally:
            B.of_grid_destroy(h)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    ref = O.poisson_solve(rho, g)
    assert np.abs(out[0][0] - ref).max() <= 1e-9 * np.abs(ref).max()
    ref = O.kernel_solve(rho, g, kf2, P, Q)
    assert np.abs(out[0][1][..., 0] + 1j * out[0][1][..., 1] - ref).max() <= 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("low", [0.0, 0.01])
def test_v_cycle_preconditioned_nlcg(low):
    # ions along the long axis; two handles, ten and thirty steps
    M = 36
    R = np.stack([np.full(M, 1.9), np.full(M, 1.9), (np.arange(M) + 0.5) * (L3[2] / M)], -1)
    sysd = B.make_system(R + W.random_field((1, M, 3), seed=4)[0] * 0.1, np.full(M, 3.0), 1.2, 6.0)

    def run(steps):
        h = B.of_grid_create(N3, L3, 6, torch.cuda.current_stream())
        try:
            o = B.of_default_scf_opts()
            o.precision, o.nlcg_max_iter = B.OF_F32, steps
            o.nlcg_precond_shift, o.nlcg_precond_low = 1.5, low
            u = torch.ones(N3[::-1], dtype=torch.float64, device="cuda")
            B.of_profile_enable(h, 1)
            res = B.of_scf_ground_state(h, sysd, Fn.tfw(), o, u, torch.zeros_like(u), allow=(B.OF_ENOCONV,))
            ran = _launched(h)
            # outside of the solves' graphs: ten smoothing steps per V-cycle, the second shift's sweep
            assert ran["mg_smooth"] >= 10 * steps * (2 if low else 1) and "fft_direct_solve" not in ran, ran
            assert (ran.get("stencil_f32", 0) >= steps) == (low > 0.0), ran
            return res, u.cpu().numpy()
        finally:
            B.of_grid_destroy(h)

    few, _ = run(10)
    more, u = run(30)
    again, v = run(30)
    assert np.array_equal(u, v) and more.energy == again.energy
    assert np.isfinite(u).all() and more.energy < few.energy and more.nlcg_residual < few.nlcg_residual
