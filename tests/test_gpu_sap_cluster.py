"""The cluster SAP kernel's half spinors on the faces between domains: M_SAP is
bit for bit that of the one-CTA kernel for faces that fill the halo buffer
exactly (extents of two), for extents of one whose faces do not fit it (the
neighbours' x is then read in place), for two domains in a direction (both
faces towards the same domain), both time boundaries and several right-hand
sides."""

import numpy as np
import pytest

from gpu_util import Problem, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,sdom,bc_t", [
    ((8, 4, 4, 4), (2, 2, 2, 2), -1), ((12, 4, 4, 4), (3, 2, 1, 2), -1), ((8, 4, 4, 4), (2, 1, 1, 2), 1),
    ((12, 20, 4, 6), (6, 5, 2, 3), 1), ((8, 8, 8, 16), (4, 2, 4, 8), -1), ((32, 12, 8, 6), (16, 6, 4, 3), -1)])
def test_cluster_halo_matches_one_cta_kernel(dims, sdom, bc_t):
    from paper_2109_10687_gb300 import binding as B
    p = Problem(dims, (2, 2, 2, 1), eps=0.3, kappa=0.12, csw=1.0, seed=1161, bc_t=bc_t, oracle=False)
    try:
        B.qcd_set_sap_domain(p.lat.ctx, sdom)
        srcs = np.stack([p.source(2170 + r) for r in range(2)])
        for n_sap, n_jac in ((0, 1), (1, 2), (3, 4)):
            out = []
            for shape in (0, 1):
                B.qcd_set_sap_shape(p.lat.ctx, shape)
                out.append(to_np(p.lat.sap(srcs, n_sap, n_jac, "half_gauge", nrhs=2)))
            assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1]), (n_sap, n_jac)
    finally:
        p.close()
