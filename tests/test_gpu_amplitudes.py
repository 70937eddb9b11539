"""V_TF + V_xc from the amplitude, over its whole range: the density floor's side, both sides of r_s
= 1, very large values, either sign.

A grid with spacings of 10^7 bohr takes the Laplacian out of H u (1e-13 of the potential's part and
less at 2 % variation), so that H u / u is the potential.  Tolerance: each of V_TF, V_x and V_c is a
product of at most eight factors rounded to 2^-53 and known to 2^-53 themselves, the oracle's as
much again: 32 2^-53 = 3.6e-15 of the sum of their sizes; the Laplacian's part is added to it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import functional as OF  # noqa: E402
from paper_1412_8250_gb300 import binding as B, functionals as Fn  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1e-14, 3e-12, 2e-11, 1e-8, 1e-4, 0.03, 0.17, 0.4885, 0.4887, 0.9, 30.0, 1e5])
@pytest.mark.parametrize("sign", [1, -1])
def test_potential_of_amplitude(size, sign):
    n, step = (16, 15, 14), 1e7
    h = B.of_grid_create(n, tuple(step * m for m in n), 6, torch.cuda.current_stream())
    try:
        rng = np.random.default_rng(3)
        u = sign * size * rng.uniform(0.98, 1.02, n[::-1])
        hu = torch.empty(u.shape, dtype=torch.float64, device="cuda")
        zero = torch.zeros_like(hu)
        B.of_hamiltonian_apply(h, Fn.tfw(), torch.tensor(u, device="cuda"), zero, None, hu)
        rho = u * u
        vtf, vxc = OF.tf_potential(rho), OF.v_xc(rho)
        # below u^2 = 1e-30 the Thomas-Fermi part (1e-20 and less) is left out
        vtf = np.where(rho > 1e-30, vtf, 0.0)
        got = hu.cpu().numpy() / u
        scale = np.abs(vtf) + 3.0 * np.abs(vxc)   # V_x and V_c have one sign, |V_c| < |V_xc|
        assert np.all(np.abs(got - vtf - vxc) <= 3.6e-15 * scale + 20.0 / step ** 2)
    finally:
        B.of_grid_destroy(h)
