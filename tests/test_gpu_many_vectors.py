"""mg_apply on more vectors than a launch's grid has rows (65535).

Seven vectors repeated: every copy gets the same bits, and they are the
one-vector result to FP64 rounding.
"""
import numpy as np
import pytest

from gpu_common import TOL64, lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["D", "DR", "DR_DAG"])
def test_more_than_65535_vectors(op):
    lib_built()
    torch = pytest.importorskip("torch")
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    dims, n = (2, 2, 2, 2), 65535 + 8
    seven = I.gaussian_source(dims, 512, nrhs=7)
    x = torch.from_numpy(seven).cuda()[torch.arange(n, device="cuda") % 7].contiguous()
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 511))
        S.set_clover(1.0, 0.1)
        got = S.apply(getattr(B, "MG_OP_" + op), x, nrhs=n)
        one = S.apply(getattr(B, "MG_OP_" + op), np.ascontiguousarray(seven[6]))
    assert torch.equal(got, got[:7][torch.arange(n, device="cuda") % 7])
    assert rel(got[6].cpu().numpy(), one) <= TOL64
