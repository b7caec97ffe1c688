"""The TMA-fed sweep's two tile shapes, and copy boxes larger than the level,
against plain-load sweeps inside the solve (GPU): both are the same arithmetic
in the same order, so the solutions are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_1008_2801_gb300 import BatchSolver, Solver, inputs

pytestmark = pytest.mark.gpu


# 32 x 16 tiles: one column of them, part-filled rows, a part-filled column;
# 64 x 8 tiles on the last two; planes that the chunks do not divide
@pytest.mark.parametrize("n", [(32, 64, 64), (96, 48, 80), (160, 40, 72), (24, 104, 64),
                               (128, 64, 56), (64, 8, 96)])
def test_tile_shapes(cuda_device, n):
    d = inputs.stellar(n, 37)
    out = []
    for tma in (True, False):
        with Solver(d["f"].shape, d["dx"], precision="mixed", smoother="fused", tma=tma,
                    device=cuda_device) as s:
            s.set_beta(torch.from_numpy(d["beta"]).to(cuda_device))
            phi, st = s.solve(torch.from_numpy(d["f"]).to(cuda_device), tol=1e-10)
            assert st["status"] == "ok"
            assert s.smoother_kind(0) == ("fused_tma" if tma else "fused")
            out.append((phi.cpu().numpy(), st["hist"]))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]


@pytest.mark.parametrize("sizes", [(16, 24, 32, 48), (32, 48, 64, 96)])
def test_uneven_boxes(cuda_device, sizes):
    d = inputs.batched(40, 19, sizes=sizes, dx=1 / 64)
    shapes = [tuple(int(v) for v in n[::-1]) for n in d["dims"]]
    out = []
    for tma in (True, False):
        s = BatchSolver(shapes, d["dx"], precision="mixed", smoother="fused", tma=tma,
                        device=cuda_device)
        s.set_beta(s.pack([torch.from_numpy(b).to(cuda_device) for b in d["beta"]]))
        phi, st = s.solve(s.pack([torch.from_numpy(f).to(cuda_device) for f in d["f"]]), tol=1e-10)
        assert all(x["status"] == "ok" for x in st)
        out.append(phi.cpu())
        s.close()
    assert torch.equal(out[0], out[1])
