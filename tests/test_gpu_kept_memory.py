"""Device memory that a context keeps between calls.

* A call that needs more than a context keeps gives its buffers back.
* What is kept makes room for a later call that would not fit beside it.
"""
import pytest

from gpu_common import lib_built
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (16, 16, 16, 16)
VEC = 16**4 * 12 * 16          # bytes of a vector
GIB = 1 << 30


def _free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _apply(S, B, torch, n):
    x = torch.ones((n,) + DIMS[::-1] + (4, 3), dtype=torch.complex128, device="cuda")
    S.apply(B.MG_OP_D, x, nrhs=n)


def test_kept_memory_is_bounded_and_given_back():
    lib_built()
    torch = pytest.importorskip("torch")
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    with Solver(DIMS) as S:
        S.load_gauge(I.make_gauge(DIMS, 0.3, 0, 0.5, 711))
        S.set_clover(1.0, 0.1)
        S.set_params(levels=2, blocks=[(4, 4, 4, 4)], nv=[24], setup_iters=1, seed=713)
        _apply(S, B, torch, 1)
        before = _free(torch)
        _apply(S, B, torch, 400)             # 5 GB packed in, 5 GB out: more than is kept
        assert before - _free(torch) <= GIB // 4
        n = 300                              # 7.5 GB: kept
        _apply(S, B, torch, n)
        kept = before - _free(torch)
        assert 2 * n * VEC * 0.9 <= kept <= 8 * GIB
        # the setup takes 0.6 GB for null vectors, P and their orthonormalisation alone
        hold = torch.empty(_free(torch) - 3 * GIB // 8, dtype=torch.uint8, device="cuda")
        S.setup()
        eta = I.gaussian_source(DIMS, 714)
        _, info = S.solve(eta, 1e-8)
        assert info.true_residual <= 1e-8
        del hold
