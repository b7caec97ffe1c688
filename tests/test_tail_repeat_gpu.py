"""The coarse V-cycle's cluster kernel where its stages' order hangs on a
barrier: repeated solves give the same bits (GPU).

A stage that overtakes another changes the iterate, and the number of repeats
gives it room to; every sum of the solver is taken in a fixed order, so nothing
else differs between two solves.
"""
import numpy as np
import pytest
import torch

from paper_1008_2801_gb300 import BatchSolver, Solver, inputs

pytestmark = pytest.mark.gpu

REPEATS = 50


def _same(solve):
    first, st0 = solve()
    first = first.clone()
    for _ in range(REPEATS - 1):
        phi, st = solve()
        assert torch.equal(phi, first) and st == st0
    return first


def _histories(st):
    return [(x["status"], x["cycles"], x["hist"]) for x in (st if isinstance(st, list) else [st])]


# boxes whose finest level runs in the kernel: each cycle there starts from the
# iterate, which is copied over the zeros that other threads wrote
@pytest.mark.parametrize("shape,kw", [((8, 8, 8), dict()), ((16, 16, 16), dict(precision="mixed")),
                                      ((16, 16, 16), dict(coarse_cells=4096)),
                                      ((8, 8, 8), dict(bc="PPPPDD")),
                                      ((8, 8, 8), dict(krylov=True))],
                         ids=["fp64", "mixed", "split", "periodic", "krylov"])
def test_box_that_starts_in_the_kernel(cuda_device, shape, kw):
    nz, ny, nx = shape
    d = inputs.stellar((nx, ny, nz), 41)
    f = torch.from_numpy(d["f"]).to(cuda_device)
    with Solver(shape, d["dx"], device=cuda_device, **kw) as s:
        s.set_beta(torch.from_numpy(d["beta"]).to(cuda_device))

        def solve():
            phi, st = s.solve(f, tol=1e-10)
            return phi, _histories(st)

        _same(solve)


@pytest.mark.parametrize("precision,small", [("fp64", 8), ("mixed", 16)])
def test_batch_with_a_box_that_starts_in_the_kernel(cuda_device, precision, small):
    # one such box among boxes whose coarse levels start from zero; every box is
    # solved independently, so its bits are those of a batch without the others
    dims = [(64, 64, 64), (small,) * 3, (32, 64, 48), (64, 64, 64)]
    data = [inputs.stellar(n, 43 + i) for i, n in enumerate(dims)]

    def batch(which):
        shapes = [tuple(int(v) for v in dims[i][::-1]) for i in which]
        s = BatchSolver(shapes, 1 / 64, precision=precision, device=cuda_device,
                        inner_cycles=2)   # (the adaptive count is one of the whole batch)
        s.set_beta(s.pack([torch.from_numpy(data[i]["beta"]).to(cuda_device) for i in which]))
        f = s.pack([torch.from_numpy(data[i]["f"]).to(cuda_device) for i in which])

        def solve():
            phi, st = s.solve(f, tol=1e-10)
            return phi, _histories(st)

        phi = _same(solve)
        out = [a.cpu().numpy() for a in s.unpack(phi)]
        s.close()
        return out

    together, small_alone, large = batch([0, 1, 2, 3]), batch([1, 1, 1, 1]), batch([0, 2, 3])
    assert np.array_equal(together[1], small_alone[0])
    for i, a in zip((0, 2, 3), large):
        assert np.array_equal(together[i], a)


@pytest.mark.parametrize("shape", [(64, 64, 64), (64, 48, 80)])
@pytest.mark.parametrize("kw", [dict(nu1=0, nu2=3), dict(nu1=0, nu2=2, bc="PPPPDD")],
                         ids=["walls", "periodic"])
def test_no_pre_smoothing_over_two_split_levels(cuda_device, shape, kw):
    # the last split level's residuals go to the first CTA's scratch, which that
    # CTA read for the level above.  Without pre-smoothing every child is
    # restricted in both forms, so the launches give the same bits too (whether
    # or not such a cycle gets to the tolerance: two sweeps on a periodic box
    # barely converge).
    nz, ny, nx = shape
    d = inputs.stellar((nx, ny, nz), 47)
    beta, f = (torch.from_numpy(d[k]).to(cuda_device) for k in ("beta", "f"))
    with Solver(shape, d["dx"], device=cuda_device, coarse_cells=-1, **kw) as s:
        s.set_beta(beta)
        ref, want = s.solve(f, tol=1e-10)
    with Solver(shape, d["dx"], device=cuda_device, **kw) as s:
        s.set_beta(beta)

        def solve():
            phi, st = s.solve(f, tol=1e-10)
            assert _histories(st) == _histories(want)
            return phi, _histories(st)

        assert torch.equal(_same(solve), ref)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_boxes_that_stop_at_different_cycles(cuda_device, precision):
    # a box that is done leaves the kernel with its weights' copies in flight
    # while the others run; each box's bits are those of its own solve
    d = inputs.batched(24, 53, sizes=(16, 24, 32, 48), dx=1 / 48)
    shapes = [tuple(int(v) for v in n[::-1]) for n in d["dims"]]

    def batch(which):
        s = BatchSolver([shapes[i] for i in which], d["dx"], precision=precision,
                        device=cuda_device, inner_cycles=2)
        s.set_beta(s.pack([torch.from_numpy(d["beta"][i]).to(cuda_device) for i in which]))
        f = s.pack([torch.from_numpy(d["f"][i]).to(cuda_device) for i in which])

        def solve():
            phi, st = s.solve(f, tol=1e-10)
            return phi, _histories(st)

        phi, cycles = _same(solve), [c for _, c, _ in solve()[1]]
        out = [a.clone() for a in s.unpack(phi)]
        s.close()
        return out, cycles

    together, cycles = batch(range(24))
    if precision == "fp64":
        assert len(set(cycles)) > 1
    for i in range(0, 24, 5):
        alone, _ = batch([i])
        assert torch.equal(together[i], alone[0])
