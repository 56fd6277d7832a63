"""The timed choice of the batched coarsest solver is kept per Nc: two hierarchies
of one coarse lattice, two sources each, write a line each to the cache file."""
import os
import subprocess
import sys

import pytest

from gpu_common import lib_built

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child():
    from paper_1011_2775_gb300 import inputs as I
    from paper_1011_2775_gb300.solver import Solver
    dims = (8, 8, 8, 8)
    eta = I.gaussian_source(dims, 82, nrhs=2)
    with Solver(dims) as S:
        S.load_gauge(I.make_gauge(dims, 0.3, 1, 0.5, 81))
        S.set_clover(1.0, 0.1)
        for nv in (4, 12):
            S.set_params(levels=2, blocks=[(4, 4, 4, 4)], nv=[nv], seed=83)
            S.setup()
            S.solve(eta, 1e-8)


def test_choice_per_nc(tmp_path):
    lib_built()
    path = tmp_path / "choices.txt"
    env = dict(os.environ, MGCLOVER_TUNE_CACHE=str(path), PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    p = subprocess.run([sys.executable, "-c", "import test_gpu_tune_key as t; t._child()"], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    keys = [l.split()[0] for l in path.read_text().splitlines()]
    assert keys.count("coarse_group.8") == 1 and keys.count("coarse_group.24") == 1
    assert "coarse_group" not in keys
