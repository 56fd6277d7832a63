"""The streamed coarsest-level solver against the single-system kernel.

Cycles without smoothing (so the coarsest solve decides the result), the
coarse systems solved to 1e-6 by coarse_impl 3 and by coarse_impl 1: every
number of rows per item and warps per block, row counts that are not multiples
of the item, even-odd lattices and ones with an odd extent, FP32 and 16-bit
links, blocks without items, one coarse site, a restart length short enough to
restart, and a zero right-hand side.  Both solutions have a residual of 1e-6
relative; they agree to 1e-4 as the cycle parity tests ask.
"""
import numpy as np
import pytest

from gpu_common import lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # dims, block, nv, storage, restart
    ((8, 8, 8, 16), (4, 4, 4, 4), 24, 0, 64),
    ((8, 8, 8, 16), (4, 4, 4, 4), 24, 2, 16),
    ((16, 8, 8, 16), (2, 2, 2, 2), 9, 1, 64),
    ((4, 8, 4, 8), (2, 2, 2, 2), 1, 0, 64),
    ((8, 4, 8, 8), (2, 2, 2, 2), 3, 1, 64),
    ((8, 8, 8, 8), (4, 4, 4, 2), 32, 0, 64),
    ((8, 8, 8, 8), (4, 4, 4, 2), 32, 1, 16),
    ((8, 8, 16, 16), (2, 2, 2, 2), 32, 0, 64),
    ((12, 8, 8, 8), (4, 4, 4, 4), 24, 0, 64),      # 3 x 2 x 2 x 2: no even-odd
    ((12, 8, 4, 8), (4, 4, 2, 4), 7, 1, 4),
    ((12, 12, 12, 24), (4, 4, 4, 4), 24, 2, 16),
    ((12, 8, 8, 8), (4, 4, 4, 4), 32, 0, 64),
    ((4, 4, 4, 4), (4, 4, 4, 4), 8, 0, 64),        # one coarse site
]


@pytest.mark.parametrize("dims,block,nv,storage,restart", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_streamed_matches_the_single_system_kernel(dims, block, nv, storage, restart):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(dims, 0.3, 1, 0.5, 191)
    r = I.gaussian_source(dims, 192)
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.1)
        S.set_params(levels=2, blocks=[block], nv=[nv], storage=storage, nu_post=0, tol_coarse=1e-6, maxit_coarse=400,
                     restart_coarse=restart, setup_iters=1, seed=193)
        S.setup()
        S.set_params(coarse_impl=1)
        ref = S.apply(B.MG_OP_CYCLE, r)
        S.set_params(coarse_impl=3)
        got = S.apply(B.MG_OP_CYCLE, r)
        assert rel(got, ref) <= 1e-4
        assert (S.apply(B.MG_OP_CYCLE, np.zeros_like(r)) == 0).all()
        assert np.array_equal(S.apply(B.MG_OP_CYCLE, r), got)
