"""GPU operator applications with kept buffers, and the launch shapes by lattice size.

The buffers of mg_apply outlive a call: what an earlier application left in
them (here non-finite values, another operator, another number of vectors)
must not reach a later one, and the operators that write even sites only
return exact zeros on the odd ones.  The one-site-per-thread kernels take CTAs
of 32, 64 or 128 sites by lattice size; the last case is in the largest class.
Tolerances as the other operator parity tests.
"""
import numpy as np
import pytest

from gpu_common import TOL32, TOL64, lib_built, rel
from oracle.dirac import WilsonClover
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("op", ["DR", "BR", "DR_DAG"])
def test_even_site_operators_after_non_finite_input(op, prec, nrhs):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    dims = (6, 4, 2, 10)
    U = I.make_gauge(dims, 0.3, 0, 0.5, 81)
    x = I.gaussian_source(dims, 82, nrhs=nrhs)
    W = WilsonClover(U, 1.0, 0.1)
    code = getattr(B, "MG_OP_" + op)
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.1)
        fresh = S.apply(code, x, prec=prec, nrhs=nrhs)
        S.apply(B.MG_OP_D, np.full_like(np.concatenate([x, x]), np.nan), prec=prec, nrhs=2 * nrhs)
        got = S.apply(code, x, prec=prec, nrhs=nrhs)
    assert np.array_equal(fresh, got)
    odd = np.broadcast_to(~(W.even[..., 0].astype(bool)), W.shape)
    assert (got[:, odd] == 0).all()
    if op != "DR_DAG":
        f = W.b_r if op == "BR" else (lambda v: W.Dr(v * W.even))
        for q in range(nrhs):
            ref = f(x[q].reshape(W.shape + (12,))).reshape(x[q].shape)
            assert rel(got[q], ref) <= (TOL32 if prec else TOL64)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (6, 4, 8, 10), (16, 16, 8, 16), (16, 16, 32, 32)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("op", ["D", "HOP", "DP", "DR"])
def test_launch_shapes(dims, op):
    lib_built()
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.random_gauge(dims, 0.4, 83)
    x = I.gaussian_source(dims, 84)
    W = WilsonClover(U, 1.0, 0.1)
    f = {"D": W.D, "HOP": W.hop, "DP": W.Dp, "DR": lambda v: W.Dr(v * W.even)}[op]
    ref = f(x.reshape(W.shape + (12,))).reshape(x.shape)
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.0, 0.1)
        assert rel(S.apply(getattr(B, "MG_OP_" + op), x, prec=B.MG_FP64), ref) <= TOL64
        assert rel(S.apply(getattr(B, "MG_OP_" + op), x, prec=B.MG_FP32), ref) <= TOL32
