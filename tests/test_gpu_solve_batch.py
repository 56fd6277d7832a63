"""mg_solve_batch on contexts that each have a stream of their own.

The coarsest solves of the contexts are whole-GPU cooperative grids or one
launch shared by several lattices; whichever a context takes, its solutions
reach the tolerance with the oracle's D of its lattice.
"""
import numpy as np
import pytest

from gpu_common import lib_built
from oracle.dirac import WilsonClover, norm2
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# dims, block, nv, eps, m0, seed; the last has an odd coarse extent
LATTICES = [((8, 8, 8, 8), (2, 2, 2, 2), 8, 0.3, -0.1, 8101),
            ((8, 8, 8, 16), (4, 4, 4, 4), 12, 0.3, -0.1, 8102),
            ((6, 4, 4, 8), (2, 2, 2, 2), 8, 0.4, -0.15, 8103)]


# sources per context, coarse_impl
@pytest.mark.parametrize("nrhs,impl", [((3, 2, 2), 0), ((1, 1, 1), 0), ((3, 2, 2), 2)],
                         ids=["shared_launch", "a_launch_each", "forced_shared"])
def test_contexts_on_their_own_streams(nrhs, impl):
    lib_built()
    torch = pytest.importorskip("torch")
    from paper_1011_2775_gb300.solver import Solver, solve_batch
    solvers, etas, ops, streams = [], [], [], []
    for (dims, blk, nv, eps, m0, seed), n in zip(LATTICES, nrhs):
        U = I.make_gauge(dims, eps, 1, 0.5, seed)
        streams.append(torch.cuda.Stream())
        S = Solver(dims, stream=streams[-1].cuda_stream)
        S.load_gauge(U)
        S.set_clover(1.0, m0)
        S.set_params(levels=2, blocks=[blk], nv=[nv], seed=seed + 1, maxit_fine=2000, coarse_impl=impl)
        S.setup()
        solvers.append(S)
        etas.append(I.gaussian_source(dims, seed + 2, nrhs=n).reshape((n,) + dims[::-1] + (4, 3)))
        ops.append(WilsonClover(U, 1.0, m0))
    outs, infos = solve_batch(solvers, etas, 1e-10)
    for eta, psi, W, info in zip(etas, outs, ops, infos):
        for q in range(eta.shape[0]):
            res = eta[q].reshape(W.shape + (12,)) - W.D(psi[q].reshape(W.shape + (12,)))
            assert np.sqrt(norm2(res) / norm2(eta[q])) <= 1e-10
        assert info.coarse_iterations[1] > 0
    for S in solvers:
        S.close()
