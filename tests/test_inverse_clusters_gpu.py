"""The dense coarsest inverse by clusters of 16, 8, 4, 2 CTAs and by one (GPU).

More boxes take smaller clusters, as a device that cannot hold the larger ones
does.  A row's updates keep their order whatever the number of CTAs, so box 0's
solution has the same bits in every batch.
"""
import pytest
import torch

from paper_1008_2801_gb300 import BatchSolver, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [(16, 16, 6), (14, 10, 6)])   # (nx, ny, nz): 192 and 105 cells
def test_inverse_keeps_its_bits(cuda_device, precision, n):
    d = inputs.stellar(n, 67)
    beta, f = (torch.from_numpy(d[k]).to(cuda_device) for k in ("beta", "f"))
    ref = None
    for nbox in (1, 19, 38, 76, 152, 305):
        s = BatchSolver([tuple(f.shape)] * nbox, d["dx"], precision=precision, device=cuda_device,
                        inner_cycles=2)
        s.set_beta(beta.reshape(-1).repeat(nbox))
        phi, st = s.solve(f.reshape(-1).repeat(nbox), tol=1e-10)
        assert all(x["status"] == "ok" for x in st)
        got = phi[:f.numel()].clone()
        s.close()
        ref = got if ref is None else ref
        assert torch.equal(got, ref)
