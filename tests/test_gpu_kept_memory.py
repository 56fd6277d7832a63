"""Device memory that a context keeps between calls.

* A call that needs more than a context keeps gives its buffers back.
* What is kept makes room for a later call that would not fit beside it.

In a process of its own, which holds the rest of the device's memory meanwhile.
"""
import json
import os
import subprocess
import sys

import pytest

from gpu_common import lib_built

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIMS = (16, 16, 16, 16)
VEC = 16**4 * 12 * 16          # bytes of a vector
GIB = 1 << 30
MANY = 300                     # vectors: 7.5 GB in and out


def _child():
    import torch
    from paper_1011_2775_gb300 import binding as B, inputs as I
    from paper_1011_2775_gb300.solver import Solver

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    def apply(S, n):
        x = torch.ones((n,) + DIMS[::-1] + (4, 3), dtype=torch.complex128, device="cuda")
        S.apply(B.MG_OP_D, x, nrhs=n)

    with Solver(DIMS) as S:
        S.load_gauge(I.make_gauge(DIMS, 0.3, 0, 0.5, 711))
        S.set_clover(1.0, 0.1)
        S.set_params(levels=2, blocks=[(4, 4, 4, 4)], nv=[24], setup_iters=1, seed=713)
        apply(S, 1)
        before = free()
        apply(S, 400)                        # 5 GB packed in, 5 GB out: more than is kept
        large = before - free()
        apply(S, MANY)
        kept = before - free()
        # the setup takes 0.6 GB for null vectors, P and their orthonormalisation alone
        hold = torch.empty(free() - 3 * GIB // 8, dtype=torch.uint8, device="cuda")
        S.setup()
        _, info = S.solve(I.gaussian_source(DIMS, 714), 1e-8)
        del hold
    print("RESULT " + json.dumps({"large": large, "kept": kept, "residual": info.true_residual}))


def test_kept_memory_is_bounded_and_given_back():
    lib_built()
    pytest.importorskip("torch")
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    p = subprocess.run([sys.executable, "-c", "import test_gpu_kept_memory as t; t._child()"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    r = json.loads(p.stdout.split("RESULT ")[1])
    assert r["large"] <= GIB // 4
    assert 2 * MANY * VEC * 0.9 <= r["kept"] <= 8 * GIB
    assert r["residual"] <= 1e-8
