"""The coarse V-cycle that runs in one thread-block cluster per box against
the same levels as separate launches (GPU).

Every stage does the same arithmetic per cell in both forms, so the solutions
agree to rounding (1e-12, the bar of the existing comparison of the two).  The
shapes put the split over the cluster at its edges: as many planes as CTAs,
fewer planes than CTAs, a number they do not divide, levels just above and
below the size one CTA runs alone, a split level above an unsplit one, rows of
an odd number of pairs, and boxes that are their own coarsest level.
"""
import numpy as np
import pytest
import torch

from paper_1008_2801_gb300 import BatchSolver, Solver, inputs

pytestmark = pytest.mark.gpu


def _solve(shape, dev, precision, cells, **kw):
    nz, ny, nx = shape
    d = inputs.stellar((nx, ny, nz), 31)
    if precision == "mixed" and not kw.get("krylov"):
        kw = dict(kw, inner_cycles=2)   # (the adaptive exit may turn on a rounding)
    with Solver(shape, d["dx"], precision=precision, device=dev, coarse_cells=cells, **kw) as s:
        s.set_beta(torch.from_numpy(d["beta"]).to(dev))
        phi, st = s.solve(torch.from_numpy(d["f"]).to(dev), tol=1e-10)
        return phi.cpu().numpy(), st


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(64, 64, 64), (48, 64, 80), (16, 96, 160), (112, 24, 40),
                                   (160, 16, 16), (8, 8, 8), (2, 6, 10), (20, 20, 36)])
def test_cluster_matches_launches(cuda_device, precision, shape):
    ref, st0 = _solve(shape, cuda_device, precision, -1)
    got, st = _solve(shape, cuda_device, precision, 0)
    assert st["status"] == "ok" and st["cycles"] == st0["cycles"]
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("kw", [dict(bc="PPPPDD"), dict(bc="DDDDPP"), dict(bc="NNPPND"),
                                dict(krylov=True), dict(nu1=0, nu2=3), dict(nu1=3, nu2=0),
                                dict(full_residual=True), dict(use_graph=False),
                                dict(coarse_cells=4096)],
                         ids=lambda k: ",".join(f"{a}={b}" for a, b in k.items()))
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_cluster_options(cuda_device, precision, kw):
    kw = dict(kw)
    cells = kw.pop("coarse_cells", 0)
    ref, st0 = _solve((48, 32, 64), cuda_device, precision, -1, **kw)
    got, st = _solve((48, 32, 64), cuda_device, precision, cells, **kw)
    assert st["status"] == "ok" and st["cycles"] == st0["cycles"]
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("nbox", [3, 20, 90, 200])
def test_cluster_sizes_of_batches(cuda_device, nbox):
    # the cluster shrinks as the boxes grow in number: 16 CTAs to one
    d = inputs.batched(nbox, 17, sizes=(8, 16, 24, 32), dx=1 / 32)
    shapes = [tuple(int(v) for v in n[::-1]) for n in d["dims"]]
    out = []
    for cells in (-1, 0):
        s = BatchSolver(shapes, d["dx"], device=cuda_device, coarse_cells=cells)
        s.set_beta(s.pack([torch.from_numpy(b).to(cuda_device) for b in d["beta"]]))
        phi, st = s.solve(s.pack([torch.from_numpy(f).to(cuda_device) for f in d["f"]]), tol=1e-10)
        assert all(x["status"] == "ok" for x in st)
        out.append((phi.cpu().numpy(), [x["cycles"] for x in st]))
        s.close()
    assert out[0][1] == out[1][1]
    assert np.linalg.norm(out[1][0] - out[0][0]) <= 1e-12 * np.linalg.norm(out[0][0])


@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 5, 3), (4, 4, 3), (7, 3, 6), (8, 8, 2), (5, 9, 17),
                                   (9, 10, 11), (8, 8, 16)])
@pytest.mark.parametrize("singular", [False, True])
def test_cluster_inverse(cuda_device, shape, singular):
    # one, eight and sixteen CTAs, rows in shared memory and (1024) in scratch:
    # A Ainv against the identity, less the constant part when A is singular.
    # Backward error of an elimination without exchanges on a diagonally
    # dominant matrix: a few n eps |A| |Ainv|.
    from paper_1008_2801_gb300 import ops as K

    rng = np.random.default_rng(71)
    beta = torch.from_numpy(rng.uniform(0.5, 2.0, shape)).to(cuda_device)
    if singular and beta.numel() == 1:
        pytest.skip("A is 0")
    w = K.face_weights(beta, 1.0, bc=63 if singular else 0)
    inv = K.bottom_inverse(w, shape, singular).cpu().numpy()
    wx, wy, wz = (K.get(t, shape, k).cpu().numpy() for t, k in zip(w, "xyz"))
    n = inv.shape[0]
    idx = np.arange(n).reshape(shape)
    A = np.zeros((n, n))
    np.fill_diagonal(A, -(wx[:, :, :-1] + wx[:, :, 1:] + wy[:, :-1] + wy[:, 1:] + wz[:-1]
                          + wz[1:]).ravel())
    for a, b, v in ((idx[:, :, :-1], idx[:, :, 1:], wx[:, :, 1:-1]),
                    (idx[:, :-1], idx[:, 1:], wy[:, 1:-1]), (idx[:-1], idx[1:], wz[1:-1])):
        A[a.ravel(), b.ravel()] = v.ravel()
        A[b.ravel(), a.ravel()] = v.ravel()
    assert np.array_equal(inv, inv.T)
    eye = np.eye(n) - (1.0 / n if singular else 0.0)
    if singular:   # on zero-mean right-hand sides
        inv = inv @ eye
    bar = 8 * n * 2.0 ** -53 * np.linalg.norm(A, 1) * np.linalg.norm(inv, 1)
    assert np.abs(A @ inv - eye).max() <= bar
