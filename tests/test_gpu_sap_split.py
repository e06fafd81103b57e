"""The SAP kernel of storage blocks other than 4^4 against the oracle: domains
of less than, exactly and more than a block of 64 sites; a last block that is
not full; directions in which a domain is one site wide (every hop leaves), two
(one body for both hops) and more; one and three right-hand sides.  And the
kernel with four threads per site against the block kernel of 4^4 domains, bit
for bit."""

import numpy as np
import pytest

from gpu_util import Problem, rel_l2, to_np
from oracle import sap

pytestmark = pytest.mark.gpu

CASES = [((2, 2, 2, 2), (1, 1, 1, 1), -1), ((6, 4, 4, 2), (1, 2, 2, 1), 1), ((4, 4, 4, 8), (2, 2, 2, 2), -1),
         ((8, 8, 4, 8), (2, 4, 2, 4), 1), ((8, 4, 8, 16), (4, 2, 4, 4), -1), ((16, 8, 8, 4), (8, 4, 4, 2), -1)]


@pytest.fixture(scope="module", params=CASES, ids=lambda c: "x".join(map(str, c[0])) + "_d" + "x".join(map(str, c[1])))
def prob(request):
    dims, domain, bc_t = request.param
    p = Problem(dims, domain, eps=0.3, kappa=0.12, csw=1.0, seed=1301, bc_t=bc_t)
    yield p
    p.close()


# float16 storages against the unrounded operator; the iterates differ by the
# rounding of links, C_inv (2^-11 each) and, for half, s
@pytest.mark.parametrize("sap_prec,tol", [("single", 1e-6), ("half_gauge", 1e-3), ("half", 2e-3)])
@pytest.mark.parametrize("n_sap,n_jac", [(0, 1), (2, 3), (4, 4)])
def test_msap(prob, sap_prec, tol, n_sap, n_jac):
    srcs = np.stack([prob.source(2301 + r) for r in range(3)])
    got = to_np(prob.lat.sap(srcs, n_sap, n_jac, sap_prec, nrhs=3))
    for r in range(3):
        assert rel_l2(got[r], sap.msap(prob.op, srcs[r], n_sap, n_jac)) <= tol
    one = to_np(prob.lat.sap(srcs[1], n_sap, n_jac, sap_prec))
    assert np.array_equal(one, got[1])


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (8, 16, 8, 24)])
@pytest.mark.parametrize("sap_prec", ["single", "half_gauge", "half"])
def test_equals_the_block_kernel_on_4x4x4x4_domains(dims, sap_prec):
    from paper_2109_10687_gb300 import binding as B
    p = Problem(dims, (4, 4, 4, 4), eps=0.3, kappa=0.12, csw=1.0, seed=1302, oracle=False)
    try:
        b = p.source(2310)
        tuned = to_np(p.lat.sap(b, 3, 4, sap_prec))
        assert "4threads_per_site" in B.qcd_tuning_report(p.lat.ctx)
        B.qcd_set_sap_shape(p.lat.ctx, 0)
        assert np.array_equal(to_np(p.lat.sap(b, 3, 4, sap_prec)), tuned)
    finally:
        p.close()
