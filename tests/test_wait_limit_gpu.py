"""Short limits on device waits: a solve ends in its result or in a timeout, and
the device stays usable (GPU)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1008_2801_gb300 import MGError, Solver, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(128, 64, 64), (96, 48, 80)])   # 64- and 32-wide tiles
@pytest.mark.parametrize("limit", [1, 2, 3, 50, 2000])
def test_tile_copy_waits(cuda_device, n, limit):
    # after a consumer gave up the producer issues no further copy: no solve may
    # end in other bits than the default bound's
    d = inputs.stellar(n, 57)
    beta, f = (torch.from_numpy(d[k]).to(cuda_device) for k in ("beta", "f"))
    kw = dict(precision="mixed", smoother="fused", tma=True, device=cuda_device)
    with Solver(f.shape, d["dx"], **kw) as s:
        s.set_beta(beta)
        ref, _ = s.solve(f, tol=1e-10)
        with Solver(f.shape, d["dx"], wait_limit=limit, **kw) as q:
            q.set_beta(beta)
            for _ in range(20):
                try:
                    phi, _ = q.solve(f, tol=1e-10)
                except MGError as e:
                    assert e.name == "timeout"
                else:
                    assert torch.equal(phi, ref)
        again, _ = s.solve(f, tol=1e-10)
    assert torch.equal(again, ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_limit_on_the_cg_coarsest_solve(cuda_device, precision):
    # 13 tiles of 9 x 9 cells: one cluster by default, a limit takes the grid
    # barrier.  One poll does not see thirteen CTAs through some hundred barriers;
    # a large number does, with the default form's bits.
    d = inputs.stellar((9, 9, 13), 59)
    beta, f = (torch.from_numpy(d[k]).to(cuda_device) for k in ("beta", "f"))
    kw = dict(precision=precision, device=cuda_device)
    out = []
    for limit in (0, 1 << 20):
        with Solver(f.shape, d["dx"], wait_limit=limit, **kw) as s:
            s.set_beta(beta)
            phi, st = s.solve(f, tol=1e-10)
            assert st["status"] == "ok"
            out.append(phi)
    assert torch.equal(*out)
    with Solver(f.shape, d["dx"], wait_limit=1, **kw) as s:
        s.set_beta(beta)
        with pytest.raises(MGError) as ei:
            s.solve(f, tol=1e-10)
        assert ei.value.name == "timeout"


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape,limit", [((13, 9, 9), 0), ((13, 9, 9), 1 << 20), ((33, 33, 33), 0)])
def test_cg_around_a_cg_coarsest_solve(cuda_device, shape, limit, precision):
    # a box that is its own coarsest level: the outer iteration's solution must
    # not share an array with the inner one's residual, in either form
    nz, ny, nx = shape
    d = inputs.stellar((nx, ny, nz), 59)
    with Solver(shape, d["dx"], precision=precision, krylov=True, wait_limit=limit,
                device=cuda_device) as s:
        s.set_beta(torch.from_numpy(d["beta"]).to(cuda_device))
        phi, st = s.solve(torch.from_numpy(d["f"]).to(cuda_device), tol=1e-10)
    assert st["status"] == "ok", st
    r = O.residual(O.face_beta(d["beta"]), d["dx"], d["f"], phi.cpu().numpy())
    assert np.linalg.norm(r) <= 1.01e-10 * np.linalg.norm(d["f"])
