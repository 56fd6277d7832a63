"""D_r of an intermediate level as its smoother and solver apply it (the odd-site
links with the site inverses folded in), through the smoothing of a cycle.

With z0 the cycle of level 1 without smoothing, one minimal-residual step gives
z0 + alpha r with r = b - D_r z0, w = D_r r, alpha = <w, r> / <w, w>, and so on;
D_r here is formed in 64 bits from the coarse links.  FP32 and 16-bit links, rows
that are fewer than, equal to and more than a block's 48, multiples of 16 and not.
"""
import numpy as np
import pytest

from gpu_common import TOL32, lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)


def _dr(Y, X):
    par = (np.indices(X.shape[:4]).sum(0) % 2)[..., None]
    Xi = np.linalg.inv(X)

    def mul(M, v):
        return np.einsum("tzyxab,tzyxb->tzyxa", M, v)

    def hop(v):
        return sum(mul(Y[..., d, :, :], np.roll(v, -1 if d < 4 else 1, 3 - (d & 3))) for d in range(8))

    return lambda v: (v - hop(mul(Xi, hop(mul(Xi, v)) * par))) * (1 - par)


@pytest.mark.parametrize("storage", [0, 1, 2], ids=["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nv", [3, 7, 24, 29, 32])
def test_smoothing_applies_the_folded_operator(nv, storage):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    with Solver(DIMS) as S:
        S.load_gauge(I.make_gauge(DIMS, 0.3, 1, 0.5, 911))
        S.set_clover(1.0, 0.1)
        S.set_params(levels=3, blocks=[(2, 2, 2, 2), (2, 2, 2, 2)], nv=[nv, 6], storage=storage, setup_iters=1, seed=912,
                     nu_post=0, coarse_impl=1)
        S.setup()
        Y, X = S.coarse_links(1)
        D = _dr(Y, X)
        rng = np.random.default_rng(913)
        b = rng.standard_normal(X.shape[:5]) + 1j * rng.standard_normal(X.shape[:5])
        b = b.astype(np.complex64).astype(np.complex128)
        even = 1 - (np.indices(X.shape[:4]).sum(0) % 2)[..., None]
        z = S.apply(B.MG_OP_CYCLE, b, level=1)
        r = b * even - D(z)
        for nu in (1, 2, 3):
            w = D(r)
            alpha = np.vdot(w, r) / np.vdot(w, w)
            z = z + alpha * r
            r = r - alpha * w
            S.set_params(nu_post=nu)
            assert rel(S.apply(B.MG_OP_CYCLE, b, level=1), z) <= TOL32
