"""The float32 operators on several right-hand sides of 4^4 blocks: every result
equals the single-right-hand-side kernel's bit for bit, untuned (one per thread
on small lattices; pairs on larger ones, an odd last right-hand side included)
and tuned, on links stored as 12 and as 18 reals, for both time boundaries."""

import pytest
import torch

from gpu_util import Problem, rel_l2, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bc_t,links12,nrhs", [
    ((8, 8, 8, 8), -1, True, 2), ((8, 8, 8, 8), 1, False, 5), ((16, 8, 8, 24), -1, True, 12),
    ((16, 16, 16, 16), -1, True, 12), ((16, 16, 16, 16), 1, False, 21), ((16, 16, 8, 24), 1, True, 22)])
def test_matches_single_right_hand_side(dims, bc_t, links12, nrhs):
    from paper_2109_10687_gb300 import binding as B
    p = Problem(dims, (4, 4, 4, 4), eps=0.3, kappa=0.12, csw=1.0, seed=1401, bc_t=bc_t, oracle=dims == (8, 8, 8, 8))
    try:
        B.qcd_set_link_compression(p.lat.ctx, links12)
        assert B.qcd_link_format(p.lat.ctx) == (12 if links12 else 18)
        gen = torch.Generator("cuda").manual_seed(2401)
        srcs = torch.randn((nrhs, *p.source(1).shape), dtype=torch.complex64, device="cuda", generator=gen)
        ops = {"D": lambda v, n: p.lat.apply_D(v, "single", nrhs=n),
               "Ddag": lambda v, n: p.lat.apply_D(v, "single", dagger=True, nrhs=n),
               "A": lambda v, n: p.lat.apply_A(v, nrhs=n)}
        for tune in (False, True):
            B.qcd_set_tuning(p.lat.ctx, tune)
            for op, f in ops.items():
                got = f(srcs, nrhs)
                for r in range(nrhs):
                    assert torch.equal(got[r], f(srcs[r], 1)), (tune, op, r)
                if p.op is not None:
                    assert rel_l2(to_np(got[nrhs - 1]), getattr(p.op, op)(to_np(srcs[nrhs - 1]))) <= 1e-6
    finally:
        p.close()
