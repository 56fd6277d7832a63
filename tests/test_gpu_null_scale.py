"""Coarse links from null vectors far from unit scale.

Block Gram-Schmidt makes the same orthonormal vectors whatever the scale of the
given ones, so vectors times powers of two -- over the whole lattice, or in some
of the blocks only -- give the same coarse links, bit for bit.
"""
import numpy as np
import pytest

from gpu_common import lib_built
from oracle.philox import gaussian_vector
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _links(dims, V, storage):
    from paper_1011_2775_gb300.solver import Solver
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 311))
        S.set_clover(1.0, -0.1)
        S.set_params(levels=2, blocks=[(4, 4, 4, 4)], nv=[len(V)], storage=storage)
        S.set_null_vectors(0, V)
        S.setup()
        return S.coarse_links(1)


@pytest.mark.parametrize("storage", [0, 1], ids=["fp32", "fp16"])
def test_links_do_not_depend_on_the_scale(storage):
    lib_built()
    dims = (8, 4, 8, 8)
    shape = dims[::-1]
    V = np.stack([gaussian_vector(312, 0, k, shape, 12) for k in range(6)]).reshape((6,) + shape + (4, 3))
    V = V.astype(np.complex64).astype(np.complex128)
    ref = _links(dims, V, storage)
    W = V.copy()
    W[1] *= 2.0**-70
    W[2] *= 2.0**65
    W[3] *= 2.0**-100
    W[4] *= 2.0**100
    W[5, :4] *= 2.0**-80       # the blocks of the first four time slices
    got = _links(dims, W, storage)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
