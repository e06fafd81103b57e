"""GPU gradients of L = Re(eta^dag D^-1 b) against the float64 oracle
gradient (hopping and clover parts, raw and su(3)-projected)."""

import numpy as np
import pytest
import torch

from gpu_util import Problem, rel_l2, to_np
from oracle import grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,domain,csw", [((4, 4, 4, 4), (2, 2, 2, 2), 1.0),
                                             ((8, 8, 8, 8), (4, 4, 4, 4), 1.0),
                                             ((4, 4, 4, 8), (2, 2, 2, 2), 0.0)])
def test_grad_matches_oracle(dims, domain, csw):
    from paper_2109_10687_gb300 import binding as B
    p = Problem(dims, domain, eps=0.3, kappa=0.12, csw=csw, seed=3000)
    try:
        eta, b = p.source(3001), p.source(3002)
        lam_ref, g_ref = grad.gradients(p.op, eta, b, tol=1e-13)
        pi_ref = grad.project_su3(g_ref, p.u)
        dev = p.lat.device
        e_t = torch.view_as_real(torch.from_numpy(eta).to(dev)).contiguous()
        b_t = torch.view_as_real(torch.from_numpy(b).to(dev)).contiguous()
        gb = torch.zeros_like(b_t)
        gu = torch.zeros(p.u.shape + (2,), dtype=torch.float64, device=dev)
        params = B.qcd_solve_params_default()
        params.tol = 1e-12
        B.qcd_grad(p.lat.ctx, e_t, b_t, gb, gu, project=0, params=params)
        assert rel_l2(to_np(torch.view_as_complex(gb)), lam_ref) < 1e-9
        assert rel_l2(to_np(torch.view_as_complex(gu)), g_ref) < 1e-5
        B.qcd_grad(p.lat.ctx, e_t, b_t, None, gu, project=1, params=params)
        assert rel_l2(to_np(torch.view_as_complex(gu)), pi_ref) < 1e-5
    finally:
        p.close()


def test_autograd_function_matches_oracle():
    """torch.autograd through the library solve: L = Re(eta^dag D^-1 b),
    gradients with respect to b and U against the float64 oracle."""
    from paper_2109_10687_gb300 import binding as B
    from paper_2109_10687_gb300.autograd import solve
    p = Problem((4, 4, 4, 8), (2, 2, 2, 2), eps=0.3, kappa=0.12, csw=1.0, seed=3100)
    try:
        eta, b = p.source(3101), p.source(3102)
        lam_ref, g_ref = grad.gradients(p.op, eta, b, tol=1e-13)
        dev = p.lat.device
        bt = torch.from_numpy(b).to(dev).requires_grad_(True)
        ut = torch.from_numpy(p.u).to(dev).requires_grad_(True)
        et = torch.from_numpy(eta).to(dev)
        params = B.qcd_solve_params_default()
        params.tol = 1e-12
        x = solve(bt, ut, p.lat, 0.12, 1.0, params)
        loss = torch.sum(torch.conj(et) * x).real
        loss.backward()
        x_ref = grad.solve_D(p.op, b)
        assert abs(loss.item() - np.vdot(eta.ravel(), x_ref.ravel()).real) < 1e-9 * abs(loss.item())
        assert rel_l2(to_np(bt.grad), lam_ref) < 1e-9
        assert rel_l2(to_np(ut.grad), g_ref) < 1e-5
    finally:
        p.close()


@pytest.mark.parametrize("dims,kept", [((8, 8, 8, 16), True), ((16, 16, 16, 32), False)])
def test_scratch_beyond_the_bound_is_given_back(dims, kept):
    """Both solves and the force take 1392 B per site: 11 MB, which the context
    keeps, and 182 MB, which it does not."""
    from paper_2109_10687_gb300 import binding as B

    p = Problem(dims, (4, 4, 4, 4), eps=0.2, kappa=0.1, csw=1.0, seed=3200, oracle=False)
    try:
        vol = int(np.prod(dims))
        need = 1392 * vol
        assert (need <= 128 << 20) == kept
        b_t = torch.view_as_real(torch.from_numpy(p.source(3201, 2))).cuda().contiguous()
        x = torch.empty_like(b_t)
        gb = torch.empty_like(b_t[0])
        gu = torch.empty(p.lat.site_shape + (4, 3, 3, 2), dtype=torch.float64, device="cuda")
        params = B.qcd_solve_params_default()
        B.qcd_solve(p.lat.ctx, x, b_t, 2, params)  # the workspace and its graphs are there
        B.qcd_grad(p.lat.ctx, b_t[0], b_t[1], gb, None, x=x[1], lam=x[0], params=params)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        held = []
        for _ in range(2):
            B.qcd_grad(p.lat.ctx, b_t[0], b_t[1], gb, gu, params=params)
            held.append(before - torch.cuda.mem_get_info()[0])
        assert held[0] == held[1]  # nothing is left behind by each call
        # allocations are rounded up to 2 MB
        assert held[0] <= (need + (2 << 20) if kept else 2 << 20)
    finally:
        p.close()
