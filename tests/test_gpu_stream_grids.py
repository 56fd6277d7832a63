"""A coarse lattice whose smaller candidate grid has no plan in the streamed solver.

19 x 4 x 38 x 4 sites of Nc = 22 fit the streamed solver on the full grid; on the
88 blocks that would split its rows evenly, a block's sites leave no shared memory
for a row of links.  The choice of the coarsest solver has to pass over that grid,
and the cycle it gives solves the system as the single-system kernel's does.
"""
import pytest

from gpu_common import lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (38, 4, 38, 4)


@pytest.mark.parametrize("impl", [0, 3], ids=["chosen", "streamed"])
def test_grid_without_a_plan_is_passed_over(impl):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(DIMS, 0.3, 1, 0.5, 291)
    r = I.gaussian_source(DIMS, 292)
    with Solver(DIMS) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.1)
        S.set_params(levels=2, blocks=[(2, 1, 1, 1)], nv=[11], nu_post=0, tol_coarse=1e-6, maxit_coarse=400,
                     restart_coarse=64, setup_iters=1, seed=293)
        S.setup()
        S.set_params(coarse_impl=1)
        ref = S.apply(B.MG_OP_CYCLE, r)
        S.set_params(coarse_impl=impl)
        assert rel(S.apply(B.MG_OP_CYCLE, r), ref) <= 1e-4
