"""Thin coarsest levels solved without the coarse V-cycle's finer levels (GPU).

With coarse_cells = -1 the cluster kernel still solves the coarsest level, and
a thin one (a row of 1001 cells, 2 x 511) needs more shared memory than a kernel
may have by default.  In a process of its own: the allowance belongs to the
kernel, so an earlier solver of the process may have raised it.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
import numpy as np, torch
import oracle as O
from paper_1008_2801_gb300 import Solver, inputs
precision, shape = sys.argv[1], tuple(int(v) for v in sys.argv[2:5])
nz, ny, nx = shape
d = inputs.stellar((nx, ny, nz), 51)
with Solver(shape, d["dx"], precision=precision, coarse_cells=-1, device="cuda:0") as s:
    s.set_beta(torch.from_numpy(d["beta"]).cuda())
    phi, st = s.solve(torch.from_numpy(d["f"]).cuda(), tol=1e-10)
assert st["status"] == "ok", st
r = O.residual(O.face_beta(d["beta"]), d["dx"], d["f"], phi.cpu().numpy())
assert np.linalg.norm(r) <= 1.01e-10 * np.linalg.norm(d["f"])
"""


@pytest.mark.parametrize("precision,shape", [("fp64", (1001, 1, 1)), ("fp64", (511, 1, 2)),
                                             ("mixed", (1, 1, 1001)), ("mixed", (1023, 1, 1))])
def test_thin_coarsest_level_in_a_fresh_process(cuda_device, precision, shape):
    r = subprocess.run([sys.executable, "-c", SCRIPT, precision, *map(str, shape)], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
