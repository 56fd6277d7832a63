"""The force in passes by plane and parity, where the contributions of all
plaquettes do not fit in the memory that is left.

Against the one-pass force of the same fields on a context with room (which the
other force tests compare with the oracle): the same terms added in another order.
Isotropic and anisotropic operator, both kinds, both precisions.
"""
import pytest

from gpu_common import TOL32, TOL64, lib_built, rel
from paper_1011_2775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (16, 16, 16, 16)
MIB = 1 << 20


@pytest.mark.parametrize("fp32", [False, True], ids=["fp64", "fp32"])
@pytest.mark.parametrize("aniso", [False, True], ids=["isotropic", "anisotropic"])
def test_force_in_passes(fp32, aniso):
    lib_built()
    torch = pytest.importorskip("torch")
    from paper_1011_2775_gb300 import binding as B
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(DIMS, 0.3, 0, 0.5, 811)
    lam = torch.from_numpy(I.gaussian_source(DIMS, 812)).cuda()
    psi = torch.from_numpy(I.gaussian_source(DIMS, 813)).cuda()
    kinds = [k | (B.MG_FORCE_FP32 if fp32 else 0) for k in (B.MG_FORCE_SU3, B.MG_FORCE_WIRTINGER)]

    def run(leave):
        with Solver(DIMS) as S:
            S.load_gauge(U)
            if aniso:
                S.set_clover_aniso((0.4, 0.5, 0.6, 1.0), 1.1, 1.4, 0.1)
            else:
                S.set_clover(1.2, 0.1)
            F = [torch.zeros(DIMS[::-1] + (4, 3, 3), dtype=torch.complex128, device="cuda") for _ in kinds]
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            before = torch.cuda.mem_get_info()[0]
            hold = torch.empty(before - leave, dtype=torch.uint8, device="cuda") if leave else None
            room = torch.cuda.mem_get_info()[0]
            for f, k in zip(F, kinds):
                B.mg_force(S.ctx, f, lam, psi, k)
            kept = room - torch.cuda.mem_get_info()[0]
            del hold
            return [f.cpu().numpy() for f in F], kept

    half = 2 if fp32 else 1
    ref, kept = run(0)
    assert kept >= 280 * MIB / half          # 24 MiB of vectors, 54 of insertions, 216 of contributions
    got, kept = run(160 * MIB // half)
    assert kept <= 90 * MIB / half + 8 * MIB
    for a, b in zip(got, ref):
        assert rel(a, b) <= (TOL32 if fp32 else TOL64)
