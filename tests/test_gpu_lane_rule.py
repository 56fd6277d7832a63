"""Operators where one launch has four lanes per site and another one thread.

At 16384 sites an FP64 launch of both parities takes a thread per site and one of a
single parity four lanes; at 12^3x24 the same holds in FP32, and at 12x12x12x16 the
sites of both parities lie just above the line.  Every operator against the oracle,
and the allocation-free form gives mg_apply's bits.
"""
import numpy as np
import pytest

from gpu_common import TOL32, TOL64, lib_built, rel
from oracle.dirac import WilsonClover
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 16, 16), (12, 12, 12, 16), (12, 12, 12, 24)], ids=lambda d: "x".join(map(str, d)))
def test_operators_at_the_lines(dims):
    lib_built()
    torch = pytest.importorskip("torch")
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(dims, 0.4, 0, 0.5, 951)
    W = WilsonClover(U, 1.1, 0.05)
    x = I.gaussian_source(dims, 952)
    refs = {"D": W.D, "HOP": W.hop, "DP": W.Dp, "DR": lambda v: W.Dr(v * W.even), "BR": W.b_r}
    with Solver(dims) as S:
        S.load_gauge(U)
        S.set_clover(1.1, 0.05)
        dx = torch.from_numpy(x).cuda()
        for name, f in refs.items():
            op = getattr(B, "MG_OP_" + name)
            ref = f(x.reshape(W.shape + (12,))).reshape(x.shape)
            for prec, tol in ((B.MG_FP64, TOL64), (B.MG_FP32, TOL32)):
                got = S.apply(op, x, prec=prec)
                assert rel(got, ref) <= tol, (name, prec)
                if x.size <= 16384 * 12:
                    out = torch.empty_like(dx)
                    B.mg_apply_noalloc(S.ctx, op, out, dx, prec)
                    assert np.array_equal(out.cpu().numpy(), got), (name, prec)
