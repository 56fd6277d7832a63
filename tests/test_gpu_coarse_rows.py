"""GPU parity of the row kernel of the coarse links (hopping term of a coarse level).

A CTA takes 16 rows and a lane up to six steps of 32 column pairs before it
reads more: Nc below, at and above those sizes, in each storage format, against
the dequantised links.  Tolerance as the other FP32 parity tests.
"""
import numpy as np
import pytest

from gpu_common import TOL32, lib_built, rel
from oracle.dirac import shift
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nv", [1, 9, 24, 27])
def test_coarse_hop(nv, storage):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    dims = (8, 4, 4, 8)
    rng = np.random.default_rng(94)
    with Solver(dims) as S:
        S.load_gauge(I.random_gauge(dims, 0.3, 95))
        S.set_clover(1.0, 0.2)
        S.set_params(levels=2, blocks=[(2, 2, 2, 2)], nv=[nv], storage=storage)
        S.set_null_vectors(0, np.ascontiguousarray(I.gaussian_source(dims, 96, nrhs=nv)))
        S.setup()
        Y, X = S.coarse_links(1)
        v = rng.standard_normal(X.shape[:-1]) + 1j * rng.standard_normal(X.shape[:-1])
        got = S.apply(B.MG_OP_HOP, v, level=1)
    ref = sum(np.einsum("...ij,...j->...i", Y[..., d, :, :], shift(v, d % 4, +1 if d < 4 else -1)) for d in range(8))
    assert rel(got, ref) <= TOL32
