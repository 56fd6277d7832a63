"""Cycles on vectors that hold a NaN.

The other vectors of a batch get the bits they get without it, and a solve after
such a cycle succeeds, whichever coarsest solver runs.
"""
import numpy as np
import pytest

from gpu_common import lib_built
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("impl", [0, 1, 2, 3], ids=["chosen", "single", "batched", "streamed"])
@pytest.mark.parametrize("dims", [(8, 8, 8, 16), (12, 8, 8, 8)], ids=["even_odd", "odd_extent"])
def test_nan_stays_in_its_vector(dims, impl):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    r = I.gaussian_source(dims, 612, nrhs=4)
    bad = r.copy()
    bad[2, 0, 0, 0, 0] = np.nan     # a whole site, an even one
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 611))
        S.set_clover(1.0, 0.1)
        S.set_params(levels=2, blocks=[(4, 4, 4, 4)], nv=[8], seed=613, coarse_impl=impl)
        S.setup()
        ref = S.apply(B.MG_OP_CYCLE, r, nrhs=4)
        got = S.apply(B.MG_OP_CYCLE, bad, nrhs=4)
        for q in (0, 1, 3):
            assert np.array_equal(got[q], ref[q])
        assert not np.isfinite(got[2]).all()
        S.apply(B.MG_OP_CYCLE, np.ascontiguousarray(bad[2]))
        _, info = S.solve(np.ascontiguousarray(r[0]), 1e-8)
        assert info.true_residual <= 1e-8
