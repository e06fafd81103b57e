"""The SAP kernel of storage blocks other than 4^4 against the oracle: domains
of less than, exactly and more than a block of 64 sites; a last block that is
not full; directions in which a domain is one site wide (every hop leaves), two
(one body for both hops) and more; one and three right-hand sides.  And the
kernel with four threads per site, and whatever the tuner chooses, against the
block kernel of 4^4 domains, bit for bit."""

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


@pytest.mark.parametrize("dims,bc_t", [((8, 8, 8, 8), -1), ((8, 8, 8, 8), 1), ((8, 16, 8, 24), -1)])
@pytest.mark.parametrize("sap_prec", ["single", "half_gauge", "half"])
def test_four_threads_per_site_equal_the_block_kernel(dims, bc_t, sap_prec):
    """The kernel itself, not the tuner's choice: one and three right-hand sides,
    a closing sweep alone (n_sap 0) and with others before it."""
    from paper_2109_10687_gb300 import binding as B
    p = Problem(dims, (4, 4, 4, 4), eps=0.3, kappa=0.12, csw=1.0, seed=1302, bc_t=bc_t, oracle=False)
    ctx = p.lat.ctx
    try:
        srcs = np.stack([p.source(2320 + r) for r in range(3)])
        for n_sap, n_jac, nrhs in [(0, 1, 1), (0, 4, 3), (3, 4, 1), (3, 4, 3)]:
            b = srcs if nrhs > 1 else srcs[0]
            B.qcd_set_sap_shape(ctx, 0)
            want = to_np(p.lat.sap(b, n_sap, n_jac, sap_prec, nrhs=nrhs))
            B.qcd_set_sap_shape(ctx, -1)
            B.qcd_set_sap_split(ctx, 1)
            report = B.qcd_tuning_report(ctx)
            n0 = B.qcd_launch_count(ctx)
            got = to_np(p.lat.sap(b, n_sap, n_jac, sap_prec, nrhs=nrhs))
            # 2 (n_sap + 1) launches and the conversions of the fields: nothing was tuned
            assert B.qcd_launch_count(ctx) - n0 <= 2 * (n_sap + 1) + 2
            assert B.qcd_tuning_report(ctx) == report
            assert np.array_equal(got, want), (n_sap, n_jac, nrhs)
        B.qcd_set_sap_split(ctx, 0)
        assert np.array_equal(to_np(p.lat.sap(b, n_sap, n_jac, sap_prec, nrhs=nrhs)), want)
    finally:
        p.close()


@pytest.mark.parametrize("sap_prec", ["single", "half"])
def test_four_threads_per_site_in_the_device_side_loop(sap_prec):
    """Right-hand sides that stop at different iterations, the last of them in
    either half of one: the loop's flag ends every launch alike, and the solution
    is that of the block kernel in the loop driven by the host, bit for bit."""
    from paper_2109_10687_gb300 import binding as B
    p = Problem((8, 8, 8, 8), (4, 4, 4, 4), eps=0.3, kappa=0.12, csw=1.0, seed=1303, oracle=False)
    ctx = p.lat.ctx
    try:
        srcs = np.stack([p.source(2330), 0 * p.source(2331), p.source(2332)])
        srcs[2].reshape(-1)[1:] = 0  # a point source
        for inner_tol in (1e-2, 1e-4, 1e-5, 1e-6):
            args = dict(nrhs=3, tol=1e-10, sap_prec=sap_prec, inner_tol=inner_tol)
            B.qcd_set_sap_shape(ctx, 0)
            want, _, ref = p.lat.solve(srcs, use_graph=0, **args)
            B.qcd_set_sap_shape(ctx, -1)
            B.qcd_set_sap_split(ctx, 1)
            for _ in range(3):
                got, _, info = p.lat.solve(srcs, use_graph=2, **args)
                assert info.inner_iters == ref.inner_iters and info.outer_iters == ref.outer_iters
                assert np.array_equal(to_np(got), to_np(want))
            B.qcd_set_sap_split(ctx, -1)
    finally:
        p.close()


def test_sap_split_rejects_unknown_values():
    from paper_2109_10687_gb300 import binding as B
    p = Problem((4, 4, 4, 4), (2, 2, 2, 2), oracle=False)
    try:
        for mode in (-2, 2):
            assert B.lib().qcd_set_sap_split(p.lat.ctx, mode) == B.QCD_ERR_ARG
    finally:
        p.close()
