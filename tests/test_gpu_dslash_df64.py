"""The double-float D with the geometry of 4^4 blocks compiled in and with
strides known at run time: the residual a solve reports is within the
double-float bound of the float64 residual of its x, for storage blocks of
4^4 (neighbours in both directions different and coinciding) and of other
shapes, both time boundaries, one right-hand side and a batch.  The bound: 100
terms per component of D x, |D| <= 3, unit 2^-48, and one unit for b."""

import numpy as np
import pytest

from gpu_util import Problem, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,domain,bc_t", [
    ((16, 8, 8, 8), (4, 4, 4, 4), 1), ((8, 8, 8, 16), (4, 4, 4, 4), -1), ((8, 8, 4, 8), (2, 4, 2, 4), 1),
    ((4, 4, 4, 8), (1, 2, 2, 2), -1)])
def test_double_float_residual_by_storage_block(dims, domain, bc_t):
    p = Problem(dims, domain, eps=0.3, kappa=0.12, csw=1.0, seed=1411, bc_t=bc_t)
    try:
        b = np.stack([p.source(2411 + r) for r in range(2)])
        for n in (1, 2):
            src = b[0] if n == 1 else b
            x, rc, info = p.lat.solve(src, nrhs=n, tol=1e-10, sap_prec="single", inner_tol=1e-5)
            assert rc == 0
            got = to_np(x).reshape((n,) + b.shape[1:])
            norms = [np.linalg.norm(b[r].ravel()) for r in range(n)]
            r64 = [np.linalg.norm((b[r] - p.op.D(got[r])).ravel()) / norms[r] for r in range(n)]
            bound = max(2.0 ** -48 * (1 + 300 * np.linalg.norm(got[r].ravel()) / norms[r]) for r in range(n))
            assert max(r64) < 1e-10
            assert abs(info.true_resid - max(r64)) <= bound, n  # the largest of the right-hand sides
    finally:
        p.close()
