"""Fused post-smoothing at the launch shapes of large lattices and for several sources.

A lattice of 131072 sites of a parity runs the one-thread-per-site kernels in CTAs
of 128 (from 116736 sites on); batched cycles run the multi-source smoother for
every kind of first and last step.  The cycle with nu steps against the cycle
without smoothing followed by nu minimal-residual steps in FP64 numpy on the FP64
operator; tolerance as for the smaller lattices: 1e-5 for an FP32 application, times
3 for the norm of D_r, per step and the residual, 1e-4 for up to three steps.
"""
import numpy as np
import pytest

from gpu_common import lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs", [((16, 16, 32, 32), 1), ((16, 16, 32, 32), 2), ((4, 6, 2, 4), 3), ((8, 8, 8, 16), 5)],
                         ids=["large", "large_two", "small_three", "five"])
def test_post_smoothing(dims, nrhs):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    r = I.gaussian_source(dims, 192, nrhs=nrhs).reshape((nrhs,) + dims[::-1] + (4, 3))
    V = np.ascontiguousarray(I.gaussian_source(dims, 193, nrhs=2))
    even = (np.indices(dims[::-1]).sum(axis=0) % 2 == 0)[..., None, None]
    with Solver(dims) as S:
        S.load_gauge(I.random_gauge(dims, 0.3, 191))
        S.set_clover(1.0, 0.2)
        # one coarsest solver for single and batched cycles: both solve to the same tolerance
        S.set_params(levels=2, blocks=[(2, 2, 2, 2)], nv=[2], nu_post=0, coarse_impl=2)
        S.set_null_vectors(0, V)
        S.setup()
        Dr = lambda v: S.apply(B.MG_OP_DR, v, prec=B.MG_FP64, nrhs=nrhs)
        z = S.apply(B.MG_OP_CYCLE, r, nrhs=nrhs)
        res = r * even - Dr(z)
        for nu in (1, 2, 3):
            w = Dr(res)
            for q in range(nrhs):
                alpha = np.vdot(w[q], res[q]) / np.vdot(w[q], w[q]).real
                z[q] += alpha * res[q]
                res[q] -= alpha * w[q]
            S.set_params(nu_post=nu)
            got = S.apply(B.MG_OP_CYCLE, r, nrhs=nrhs)
            for q in range(nrhs):
                assert rel(got[q], z[q]) <= 1e-4, (nu, q)
