"""The gauge import and the clover build kernels against the oracle, where their
paths can go wrong.

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


@pytest.mark.parametrize("dims,domain", [((2, 2, 2, 2), (1, 1, 1, 1)), ((4, 4, 8, 12), (2, 1, 2, 2)),
                                         ((8, 8, 8, 8), (4, 4, 4, 4))])
@pytest.mark.parametrize("delta", [3e-13, 2e-9, 0.03, 0.5, 3.0])
def test_su3_check_reports_the_deviation(dims, domain, delta):
    """set_gauge's message gives the worst |Re| + |Im| of U^dag U - 1 and det U - 1:
    one link off by delta, in the fixed-point range and beyond it."""
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.lattice import Lattice

    u = random_su3_field(dims, 0.6, 4003)
    link = u[-1, 0, -1, 1, 2]
    link[1, 2] += delta * (1 - 0.5j)
    w = link.conj().T @ link - np.eye(3)
    det = np.linalg.det(link) - 1
    want = max((np.abs(w.real) + np.abs(w.imag)).max(), abs(det.real) + abs(det.imag))
    lat = Lattice(dims, domain, -1, "chiral")
    try:
        with pytest.raises(B.QcdError) as e:
            lat.set_gauge(u, check_tol=1e-13)
        got = float(str(e.value).split("SU(3) by ")[1].split()[0])
        # printed with four digits; the generated links are SU(3) to about 2e-15
        assert abs(got - want) <= 1e-3 * want + 4e-15
        lat.set_gauge(u, check_tol=2 * want)  # and what lies within the tolerance is taken
    finally:
        lat.close()


def _near_fields():
    """Links near the identity, near the diagonal matrices, and rough ones with
    a patch of each: (name, U, sites to compare)."""
    dims = (8, 8, 8, 8)
    everywhere = np.ones((8, 8, 8, 8), dtype=bool)
    for eps in (0.05, 0.01, 1e-3, 1e-6, 1e-9):
        yield "identity_%g" % eps, random_su3_field(dims, eps, 4006), everywhere
    theta = np.random.default_rng(4007).uniform(-1, 1, size=(8, 8, 8, 8, 4, 3))
    theta -= theta.mean(axis=-1, keepdims=True)
    near = random_su3_field(dims, 1e-5, 4008)
    yield "diagonal_1e-5", np.exp(1j * theta)[..., None] * near, everywhere
    yield "diagonal_small", np.exp(1e-6j * theta)[..., None] * np.eye(3), everywhere
    patch = random_su3_field(dims, 0.4, 4009)
    patch[2:5, 1:4, 3:6, 4:7] = random_su3_field(dims, 1e-6, 4006)[2:5, 1:4, 3:6, 4:7]
    inner = np.zeros((8, 8, 8, 8), dtype=bool)
    inner[3, 2, 4, 5] = True  # every leaf of this site lies in the patch
    yield "patch", patch, inner


@pytest.mark.parametrize("name,u,sites", list(_near_fields()), ids=lambda v: v if isinstance(v, str) else "")
def test_small_entries_of_the_clover_term_keep_their_bits(name, u, sites):
    """The off-diagonal part of 1 + C, relative to itself: products of float64
    numbers near one and small ones keep the small ones' relative accuracy
    (5e-16 measured in float64, against the oracle's own 2e-16)."""
    from oracle.dirac import clover_term
    from oracle.gamma import gamma_chiral
    from paper_2109_10687_gb300.lattice import Lattice

    c = clover_term(u, 0.125, 1.0, gamma_chiral())
    # colour-diagonal entries and the others, each relative to their own norm
    kinds = {"colour": ~np.kron(np.eye(3), np.ones((4, 4))).astype(bool),
             "spin": np.kron(np.eye(3), np.ones((4, 4)) - np.eye(4)).astype(bool)}
    lat = Lattice((8, 8, 8, 8), (4, 4, 4, 4), -1, "chiral")
    try:
        lat.set_gauge(u)
        lat.set_params(0.125, 1.0)
        lat.build_clover()
        m = np.empty(c.shape, dtype=complex)
        for j in range(12):
            psi = np.zeros(c.shape[:4] + (12,), dtype=complex)
            psi[..., j] = 1
            out = lat.apply_clover(psi.reshape(c.shape[:4] + (3, 4)), "double")
            m[..., :, j] = (out.detach().cpu().numpy() if hasattr(out, "detach") else out).reshape(c.shape[:4] + (12,))
    finally:
        lat.close()
    for kind, mask in kinds.items():
        ref = c[sites][..., mask]
        if np.abs(ref).max() > 0:
            assert np.linalg.norm(m[sites][..., mask] - ref) <= 2e-15 * np.linalg.norm(ref), (name, kind)


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("eps", [3e-37, 1e-38, 1e-41, 1e-44])
def test_float32_copies_below_the_normal_range(eps, inverse):
    """Off-diagonal entries of 1 + C and C_inv around float32's smallest normal
    number: the float32 copies are the float64 ones rounded (to 2^-24, or half
    of the smallest subnormal 2^-149)."""
    from paper_2109_10687_gb300.lattice import Lattice

    dims = (4, 4, 4, 4)
    h = (random_su3_field(dims, 1e-3, 4010) - np.eye(3)) * (1e3 * eps)
    h = (h - np.conj(np.swapaxes(h, -1, -2))) / 2  # anti-Hermitian: 1 + h is SU(3) to rounding
    lat = Lattice(dims, (2, 2, 2, 2), -1, "chiral")
    try:
        lat.set_gauge(np.eye(3) + h)
        lat.set_params(0.125, 1.0)
        lat.build_clover()
        psi = np.zeros((4, 4, 4, 4, 3, 4), dtype=complex)
        psi[..., 1, 2] = 1
        double, single = (lat.apply_clover(psi, prec, inverse=inverse) for prec in ("double", "single"))
        double, single = (a.detach().cpu().numpy() if hasattr(a, "detach") else a for a in (double, single))
    finally:
        lat.close()
    assert 0 < np.abs(double[..., 0, 2]).min() < 10 * eps
    for a, b in ((single.real, double.real), (single.imag, double.imag)):
        assert np.all(np.abs(a - b) <= 2.0**-24 * np.abs(b) + 2.0**-150)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, complex(0.1, np.nan)])
@pytest.mark.parametrize("site", [(0, 0, 0, 0), (7, 3, 2, 1)])
def test_non_finite_links_fail_the_su3_check(site, value):
    """The check refuses them at the default tolerance and at a wide one."""
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.lattice import Lattice

    u = random_su3_field((4, 4, 4, 8), 0.3, 4005)
    u[site + (2, 0, 1)] = value
    lat = Lattice((4, 4, 4, 8), (2, 2, 2, 2), -1, "chiral")
    try:
        for tol in ({}, {"check_tol": 10.0}):
            with pytest.raises(B.QcdError) as e:
                lat.set_gauge(u, **tol)
            assert e.value.code == B.QCD_ERR_ARG
        lat.set_params(0.12, 1.0)
        with pytest.raises(B.QcdError) as e:
            lat.build_clover()
        assert e.value.code == B.QCD_ERR_STATE
        lat.set_gauge(random_su3_field((4, 4, 4, 8), 0.3, 4005))  # and the context goes on
        lat.build_clover()
    finally:
        lat.close()


def test_non_finite_links_are_refused_by_the_clover_build():
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.lattice import Lattice

    u = random_su3_field((8, 8, 8, 8), 0.3, 4004)
    u[3, 2, 1, 5, 0, 1, 1] = np.nan
    lat = Lattice((8, 8, 8, 8), (4, 4, 4, 4), -1, "chiral")
    try:
        lat.set_gauge(u, check_tol=0.0)
        lat.set_params(0.12, 1.0)
        with pytest.raises(B.QcdError) as e:
            lat.build_clover()
        assert e.value.code == B.QCD_ERR_NONFINITE
    finally:
        lat.close()
