"""GPU parity of the fused fine-level post-smoothing, per lattice class and number of steps.

Up to a certain half volume the smoothing kernels take four lanes per site,
above it one thread; the first and the last step have kernels of their own.
The cycle with nu steps is compared with the cycle without smoothing followed
by nu minimal-residual steps in FP64 numpy on the FP64 operator.  Tolerance:
an FP32 application of D_r is good to 1e-5 (max-norm), every step applies it
once after the residual, and each rounding passes through D_r (norm at most 3
here): 1e-5 * 3 per step and the residual, 1e-4 for up to three steps.
"""
import numpy as np
import pytest

from gpu_common import lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [1, 2, 3])
@pytest.mark.parametrize("dims", [(4, 6, 2, 4), (16, 16, 16, 16), (24, 16, 16, 32)], ids=lambda d: "x".join(map(str, d)))
def test_post_smoothing(dims, nu):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.random_gauge(dims, 0.3, 91)
    r = I.gaussian_source(dims, 92)
    V = np.ascontiguousarray(I.gaussian_source(dims, 93, nrhs=2))
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.2)

        def cycle(n):
            S.set_params(levels=2, blocks=[(2, 2, 2, 2)], nv=[2], nu_pre=0, nu_post=n)
            S.set_null_vectors(0, V)
            S.setup()
            return S.apply(B.MG_OP_CYCLE, r, level=0)

        got, z = cycle(nu), cycle(0)
        Dr = lambda v: S.apply(B.MG_OP_DR, v, prec=B.MG_FP64)
        even = (np.indices(dims[::-1]).sum(axis=0) % 2 == 0)[..., None, None]
        res = r * even - Dr(z)
        for _ in range(nu):
            w = Dr(res)
            alpha = np.vdot(w, res) / np.vdot(w, w).real
            z = z + alpha * res
            res = res - alpha * w
    assert rel(got, z) <= 1e-4
