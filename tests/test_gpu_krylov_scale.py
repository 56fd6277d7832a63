"""BiCGStab on sources far from unit scale.

A source times a power of two has its solution times the same power: every FP64
step scales exactly and every scalar of the iteration is a ratio, so iterations
and solution repeat bit for bit as long as squared norms stay in FP64's range.
"""
import numpy as np
import pytest

from gpu_common import lib_built
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-440, -300, 300, 440])
def test_bicgstab_scales(power):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    dims = (4, 6, 4, 8)
    eta = I.gaussian_source(dims, 412)
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 411))
        S.set_clover(1.0, 0.2)
        S.set_params(levels=1, maxit_fine=500)
        ref, iref = S.solve(eta, 1e-10, B.MG_MODE_BICGSTAB)
        got, info = S.solve(eta * 2.0**power, 1e-10, B.MG_MODE_BICGSTAB)
    assert info.outer_iterations == iref.outer_iterations
    assert np.array_equal(got, ref * 2.0**power)


@pytest.mark.parametrize("power", [-20, 60])
def test_mixed_precision_scales(power):
    """The same for the FP32 inner solver: at 2^60 a block's sums of squares leave FP32's range."""
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    dims = (4, 6, 4, 8)
    eta = I.gaussian_source(dims, 414)
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 413))
        S.set_clover(1.0, 0.2)
        S.set_params(levels=1, maxit_fine=500)
        ref, iref = S.solve(eta, 1e-8, B.MG_MODE_BICGSTAB_MP)
        got, info = S.solve(eta * 2.0**power, 1e-8, B.MG_MODE_BICGSTAB_MP)
    assert info.outer_iterations == iref.outer_iterations
    assert np.array_equal(got, ref * 2.0**power)
