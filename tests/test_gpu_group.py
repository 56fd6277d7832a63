"""The grouped coarsest-level solver against the single-system kernel.

Cycles without smoothing (so the coarsest solve decides the result), the
coarse systems solved to 1e-6: the grouped kernel on 1 to 16 right-hand sides
-- every padded group size, with and without idle lanes of systems -- against
the single-system kernel (coarse_impl 1) on the same vectors, for even-odd
coarse lattices and ones with an odd extent, FP32 and 16-bit links, row counts
that are not multiples of the kernel's item, one zero right-hand side among
the others, and a restart length short enough to restart.  Both solutions have
a residual of 1e-6 relative; they agree to 1e-4 as the cycle parity tests ask.

The grouped kernel is chosen by the autotuner's cache file, written here in
advance and read by a fresh process; the file must come back unchanged, or the
choice was made by timing instead.
"""
import json
import os
import subprocess
import sys

import pytest

from gpu_common import lib_built

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# dims, block, nv, storage, right-hand sides, restart
CASES = [
    ((8, 8, 8, 8), (4, 4, 4, 4), 24, 0, 1, 64),
    ((8, 8, 8, 8), (4, 4, 4, 4), 24, 1, 12, 64),
    ((8, 8, 8, 16), (4, 4, 4, 4), 24, 2, 16, 64),
    ((8, 8, 8, 8), (2, 4, 4, 4), 9, 0, 5, 16),
    ((4, 4, 8, 8), (2, 2, 2, 2), 3, 0, 2, 64),
    ((4, 8, 4, 8), (2, 2, 2, 2), 1, 1, 3, 64),
    ((8, 4, 8, 12), (2, 2, 2, 2), 32, 0, 13, 16),
    ((12, 8, 8, 8), (4, 4, 4, 4), 24, 0, 1, 64),      # 3 x 2 x 2 x 2: no even-odd
    ((12, 8, 4, 8), (4, 4, 2, 4), 7, 1, 4, 16),
    ((12, 12, 8, 8), (4, 4, 4, 4), 16, 2, 9, 64),
    ((4, 4, 4, 4), (4, 4, 4, 4), 8, 0, 2, 64),        # one coarse site
]


def _child():
    import numpy as np
    from paper_1011_2775_gb300 import binding as B, inputs as I
    from paper_1011_2775_gb300.solver import Solver
    out = []
    for dims, block, nv, store, nb, restart in CASES:
        U = I.make_gauge(dims, 0.3, 1, 0.5, 91)
        r = I.gaussian_source(dims, 92, nrhs=nb)
        if nb > 3:
            r[nb // 2] = 0.0
        with Solver(dims) as S:
            S.load_gauge(U)
            S.set_clover(1.0, 0.1)
            S.set_params(levels=2, blocks=[block], nv=[nv], storage=store, nu_post=0, tol_coarse=1e-6, maxit_coarse=400,
                         restart_coarse=restart, setup_iters=2, seed=93)
            S.setup()
            S.set_params(coarse_impl=1)
            ref = np.stack([S.apply(B.MG_OP_CYCLE, np.ascontiguousarray(r[q])) for q in range(nb)])
            S.set_params(coarse_impl=0)
            got = S.apply(B.MG_OP_CYCLE, r if nb > 1 else np.ascontiguousarray(r[0]), nrhs=nb).reshape(ref.shape)
            again = S.apply(B.MG_OP_CYCLE, r if nb > 1 else np.ascontiguousarray(r[0]), nrhs=nb).reshape(ref.shape)
        err = [float(np.abs(got[q] - ref[q]).max() / max(np.abs(ref[q]).max(), 1e-300)) for q in range(nb)]
        out.append({"err": err, "same": bool(np.array_equal(got, again))})
    print("RESULT " + json.dumps(out))


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    lib_built()
    torch = pytest.importorskip("torch")
    gpu = torch.cuda.get_device_name(0).replace(" ", "_")
    path = tmp_path_factory.mktemp("tune") / "choices.txt"
    lines = []
    for dims, block, nv, store, nb, _ in CASES:
        c = " ".join(str(d // b) for d, b in zip(dims, block))
        lines.append(f"coarse_gcr4 {c} {2 * nv} {store} {gpu} 300 0.0" if nb == 1 else f"coarse_group {c} {nb} {store} {gpu} 0 0.0")
    path.write_text("\n".join(lines) + "\n")
    env = dict(os.environ, MGCLOVER_TUNE_CACHE=str(path), PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    p = subprocess.run([sys.executable, "-c", "import test_gpu_group as t; t._child()"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    chosen = [l for l in path.read_text().splitlines() if l.startswith(("coarse_gcr4", "coarse_group"))]
    assert chosen == lines
    return json.loads(p.stdout.split("RESULT ")[1])


@pytest.mark.parametrize("i", range(len(CASES)), ids=lambda i: f"{'x'.join(map(str, CASES[i][0]))}-nv{CASES[i][2]}-nb{CASES[i][4]}")
def test_group_matches_the_single_system_kernel(results, i):
    assert max(results[i]["err"]) <= 1e-4
    assert results[i]["same"]
