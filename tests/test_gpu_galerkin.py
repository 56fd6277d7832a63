"""GPU parity of the Galerkin coarse links (and the block Gram-Schmidt) at the edges of their kernels.

The projection takes two columns per thread, splits its threads into groups of
Nv, and sums the hops inside a block apart from those that cross a face: odd
Nv, one null vector, 32 of them, anisotropic blocks, coarse extents of one
(no faces at all) and two, and the projection from a coarse level, each
against the oracle's links from the same injected vectors.  Tolerance 1e-5
relative (max-norm) as the other FP32 parity tests: the FP32 null vectors and
hops carry about 1e-7, the projection sums in about 48 bits.
"""
import numpy as np
import pytest

from gpu_common import TOL32, lib_built, rel
from oracle.dirac import WilsonClover
from oracle.multigrid import Transfer, block_gram_schmidt, build_coarse
from oracle.philox import gaussian_vector
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # dims, blocks, nv, coarse_op
    ((4, 4, 4, 4), [(4, 4, 4, 4)], [1], 0),
    ((4, 4, 4, 8), [(4, 4, 4, 4)], [3], 0),
    ((8, 4, 4, 6), [(2, 4, 2, 3)], [5], 0),
    ((4, 8, 4, 4), [(4, 2, 4, 2)], [32], 0),
    ((4, 4, 8, 4), [(2, 2, 4, 4)], [7], 1),
    ((8, 8, 4, 8), [(2, 2, 2, 2), (2, 4, 1, 2)], [6, 9], 0),
    ((8, 8, 8, 8), [(8, 8, 8, 8)], [4], 0),   # a block too large for the Gram-Schmidt's shared memory
]


@pytest.mark.parametrize("dims,blocks,nv,op", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_coarse_links(dims, blocks, nv, op):
    lib_built()
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(dims, 0.3, 1, 0.5, 61)
    level = WilsonClover(U, 1.0, -0.1)
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, -0.1)
        S.set_params(levels=len(nv) + 1, blocks=blocks, nv=nv, coarse_op=op)
        vecs, shape, ndof = [], level.shape, 12
        for l, (b, n) in enumerate(zip(blocks, nv)):
            v = [gaussian_vector(62 + l, l, k, shape, ndof).astype(np.complex64).astype(np.complex128) for k in range(n)]
            S.set_null_vectors(l, np.ascontiguousarray(np.stack(v)))
            vecs.append(v)
            shape, ndof = tuple(s // k for s, k in zip(shape, b[::-1])), 2 * n
        S.setup()
        for l, b in enumerate(blocks):
            T = Transfer(level, b, block_gram_schmidt(level, b, vecs[l]))
            level = build_coarse(level, T, op="D" if op else "Dp")
            Y, X = S.coarse_links(l + 1)
            assert rel(X, level.X) <= TOL32
            Yref = np.moveaxis(level.Y, 0, 4)
            assert np.abs(Y - Yref).max() <= TOL32 * max(np.abs(Yref).max(), np.abs(level.X).max())
