"""The clover build kernel against the oracle, where its paths can go wrong.

1 + C and its inverse in float64 (through qcd_apply_clover) on lattices with
fewer sites than a block, with storage blocks smaller and larger than a warp,
and with the staged copies of 4^4 blocks; SU(3) links (fixed-point products),
links that are not SU(3) (float64 products), and clover coefficients large
enough to make 1 + C indefinite (pivoted inversion).
"""

import numpy as np
import pytest

from lattice_inputs import gaussian_spinor, random_su3_field

pytestmark = pytest.mark.gpu


def _rel(a, r):
    a = a.detach().cpu().numpy() if hasattr(a, "detach") else a
    return float(np.linalg.norm((a - r).ravel()) / np.linalg.norm(r.ravel()))


@pytest.mark.parametrize("dims,domain", [((2, 2, 2, 2), (1, 1, 1, 1)), ((4, 4, 4, 8), (2, 2, 2, 2)),
                                         ((4, 4, 8, 12), (2, 1, 2, 2)), ((8, 8, 8, 8), (4, 4, 4, 4)),
                                         ((16, 8, 8, 4), (8, 4, 4, 2))])
@pytest.mark.parametrize("csw,scale", [(1.0, 1.0), (9.0, 1.0), (1.0, 1.4)])
def test_clover_and_inverse(dims, domain, csw, scale):
    from oracle.dirac import CloverWilson, site_mul
    from oracle.gamma import gamma_chiral
    from paper_2109_10687_gb300.lattice import Lattice

    kappa = 0.125
    u = scale * random_su3_field(dims, 0.6, 4001)
    psi = gaussian_spinor(dims, 4002)
    op = CloverWilson(u, kappa, csw, gamma_chiral(), bc_t=-1)
    m = np.eye(12) + op.c
    eig = np.linalg.eigvalsh(m)
    if csw > 2:
        assert eig.min() < 0 < eig.max()  # indefinite somewhere: the pivoted path runs
    lat = Lattice(dims, domain, -1, "chiral")
    try:
        lat.set_gauge(u, check_tol=0.0)
        lat.set_params(kappa, csw)
        lat.build_clover()
        assert _rel(lat.apply_clover(psi, "double"), site_mul(m, psi)) <= 1e-14
        # an inverse is good to a few units of float64 rounding times the condition number
        cond = float((np.abs(eig).max(axis=-1) / np.abs(eig).min(axis=-1)).max())
        assert _rel(lat.apply_clover(psi, "double", inverse=True), op.apply_cinv(psi)) <= 2e-15 * max(10.0, cond)
        assert _rel(lat.apply_clover(psi, "single"), site_mul(m, psi)) <= 1e-6
        assert _rel(lat.apply_D(psi, "double"), op.D(psi)) <= 1e-14
    finally:
        lat.close()
