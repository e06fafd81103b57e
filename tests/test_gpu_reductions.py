"""The float32 reductions combine the threads' sums to float64 accuracy: fields
of one nonzero component per site, whose squares and sums are whole multiples of
2^-52 below 2, so that float64 holds every partial sum exactly and 48 bits do
not; a thread's own float32 sum has one nonzero term."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,domain", [((2, 2, 2, 2), (1, 1, 1, 1)), ((4, 4, 4, 6), (2, 2, 2, 1)),
                                         ((8, 8, 8, 8), (4, 4, 4, 4)), ((8, 8, 16, 24), (4, 4, 4, 4))])
def test_block_sums_keep_float64_accuracy(dims, domain):
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.lattice import Lattice

    vol, nrhs = int(np.prod(dims)), 3
    rng = np.random.default_rng(77)
    k = rng.integers(1, 4096, size=(nrhs, vol))  # k^2 fits float32
    one = rng.integers(0, vol, size=nrhs)        # the site of the entry 1
    v = k * 2.0**-26
    v[np.arange(nrhs), one] = 1.0
    w = np.where(rng.random((nrhs, vol)) < 0.5, v, -v)
    assert (v**2).sum(axis=1).max() < 2
    ints = np.rint(v * 2.0**26).astype(object)
    want = [float(sum(x * x for x in ints[r])) * 2.0**-52 for r in range(nrhs)]
    signed = [float(sum(x * y for x, y in zip(ints[r], np.rint(w[r] * 2.0**26).astype(object)))) * 2.0**-52
              for r in range(nrhs)]

    def field(lat, vals):
        psi = np.zeros((nrhs,) + tuple(reversed(dims)) + (3, 4), dtype=complex)
        psi[..., 0, 0] = vals.reshape((nrhs,) + tuple(reversed(dims)))
        return lat.to_internal(psi, "single", nrhs)

    lat = Lattice(dims, domain, -1, "chiral")
    try:
        a, b = field(lat, v), field(lat, w)
        assert B.qcd_norm2(lat.ctx, a, B.PREC_SINGLE, nrhs) == want
        assert B.qcd_norm2_noalloc(lat.ctx, a, B.PREC_SINGLE, nrhs) == want
        assert B.qcd_cdot(lat.ctx, a, b, B.PREC_SINGLE, nrhs) == signed
    finally:
        lat.close()


def test_block_sums_beyond_float32_are_taken_in_float64():
    """Squares within float32's range whose sum is not."""
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.lattice import Lattice

    dims = (4, 4, 4, 6)
    psi = np.zeros(tuple(reversed(dims)) + (3, 4), dtype=complex)
    psi[..., 0, 0] = 2.0**63.5
    psi = psi.astype(np.complex64).astype(complex)
    lat = Lattice(dims, (2, 2, 2, 1), -1, "chiral")
    try:
        got = B.qcd_norm2(lat.ctx, lat.to_internal(psi, "single"))[0]
        want = float((np.abs(psi.real.astype(np.float32)) ** 2).astype(float).sum())
        assert got > 3.5e38 and abs(got - want) <= 1e-6 * want
    finally:
        lat.close()
