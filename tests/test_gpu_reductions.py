"""GPU solves whose reductions and coefficient updates run at the edges of their grids.

Every inner product of the Krylov solvers goes through one grid-wide sum
(transposed warp sums, block sums in order, the last block's total): lattices
of less than one warp's vectors, of one ragged block, and of more blocks than
the reduction grid has, in the FP64, the mixed-precision and the
normal-equation solver.  A solution is right when the oracle's D gives back
the source to the requested residual.
"""
import numpy as np
import pytest

from gpu_common import lib_built
from oracle.dirac import WilsonClover, norm2
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 4, 2, 6), (6, 4, 8, 10), (16, 16, 8, 16)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("mode", ["BICGSTAB", "BICGSTAB_MP", "CGNR", "EO_GCR"])
def test_solve(dims, mode):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(dims, 0.3, 0, 0.5, 71)
    eta = I.gaussian_source(dims, 72)
    W = WilsonClover(U, 1.0, 0.3)
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.3)
        S.set_params(levels=1, maxit_fine=2000)
        psi, info = S.solve(eta, 1e-10, getattr(B, "MG_MODE_" + mode))
    r = eta.reshape(W.shape + (12,)) - W.D(psi.reshape(W.shape + (12,)))
    assert np.sqrt(norm2(r) / norm2(eta)) <= 1.01e-10
    assert info.true_residual <= 1e-10
