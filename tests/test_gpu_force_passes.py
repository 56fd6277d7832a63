"""The force in passes by plane and parity, where the contributions of all
plaquettes do not fit in the memory that is left.

Against the one-pass force of the same fields on a context with room (which the
other force tests compare with the oracle): the same terms added in another order.
Isotropic and anisotropic operator, both kinds, both precisions.  In a process of
its own, which holds the rest of the device's memory meanwhile.
"""
import json
import os
import subprocess
import sys

import pytest

from gpu_common import TOL32, TOL64, lib_built, rel

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIMS = (16, 16, 16, 16)
MIB = 1 << 20


def _child():
    import torch
    from paper_1011_2775_gb300 import binding as B, inputs as I
    from paper_1011_2775_gb300.solver import Solver
    U = I.make_gauge(DIMS, 0.3, 0, 0.5, 811)
    lam = torch.from_numpy(I.gaussian_source(DIMS, 812)).cuda()
    psi = torch.from_numpy(I.gaussian_source(DIMS, 813)).cuda()

    def run(aniso, kinds, leave):
        with Solver(DIMS) as S:
            S.load_gauge(U)
            if aniso:
                S.set_clover_aniso((0.4, 0.5, 0.6, 1.0), 1.1, 1.4, 0.1)
            else:
                S.set_clover(1.2, 0.1)
            F = [torch.zeros(DIMS[::-1] + (4, 3, 3), dtype=torch.complex128, device="cuda") for _ in kinds]
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            hold = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda") if leave else None
            room = torch.cuda.mem_get_info()[0]
            for f, k in zip(F, kinds):
                B.mg_force(S.ctx, f, lam, psi, k)
            kept = room - torch.cuda.mem_get_info()[0]
            del hold
            return [f.cpu().numpy() for f in F], kept

    out = {}
    for aniso in (False, True):
        for fp32 in (False, True):
            kinds = [k | (B.MG_FORCE_FP32 if fp32 else 0) for k in (B.MG_FORCE_SU3, B.MG_FORCE_WIRTINGER)]
            ref, kept = run(aniso, kinds, 0)
            got, kept_passes = run(aniso, kinds, 160 * MIB // (2 if fp32 else 1))
            out[f"{aniso}-{fp32}"] = {"kept": kept, "kept_passes": kept_passes, "rel": [rel(a, b) for a, b in zip(got, ref)]}
    print("RESULT " + json.dumps(out))


@pytest.fixture(scope="module")
def results():
    lib_built()
    pytest.importorskip("torch")
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    p = subprocess.run([sys.executable, "-c", "import test_gpu_force_passes as t; t._child()"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    return json.loads(p.stdout.split("RESULT ")[1])


@pytest.mark.parametrize("fp32", [False, True], ids=["fp64", "fp32"])
@pytest.mark.parametrize("aniso", [False, True], ids=["isotropic", "anisotropic"])
def test_force_in_passes(results, aniso, fp32):
    r = results[f"{aniso}-{fp32}"]
    half = 2 if fp32 else 1
    assert r["kept"] >= 280 * MIB / half          # 24 MiB of vectors, 54 of insertions, 216 of contributions
    assert r["kept_passes"] <= 90 * MIB / half + 8 * MIB
    assert max(r["rel"]) <= (TOL32 if fp32 else TOL64)
