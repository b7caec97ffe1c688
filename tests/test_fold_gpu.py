"""The restriction that also applies the coarse level's first red pass, and the
column kernels' depths, on shapes at the rules' edges (GPU).

The folded pass is the value the pass's FMA chain has on a zero start, so the
solution is the persistent launches' and the oracle's; the bars are those of
the tests of the two forms: 1e-12 between evaluation orders, 1e-9 against the
oracle at 1e-10.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1008_2801_gb300 import LevelSolver, MGError, Solver, inputs

pytestmark = pytest.mark.gpu


# coarse sets of 32^3 cells (not folded) and just above; one and two folded
# levels; odd numbers of pairs a row; columns of 4 and of 16 planes
@pytest.mark.parametrize("n", [(64, 64, 64), (64, 64, 72), (128, 96, 160), (80, 88, 104),
                               (256, 96, 208)])
@pytest.mark.parametrize("kw", [dict(), dict(krylov=True), dict(nu1=1, nu2=3)],
                         ids=lambda k: ",".join(f"{a}={b}" for a, b in k.items()) or "plain")
def test_folded_red_pass(cuda_device, n, kw):
    if kw.get("nu1") == 1 and n[0] > 128:
        pytest.skip("one large shape is enough")
    d = inputs.stellar(n, 23)
    beta, f = (torch.from_numpy(d[k]).to(cuda_device) for k in ("beta", "f"))
    out = []
    for persistent in (False, True):
        with Solver(f.shape, d["dx"], device=cuda_device, coarse_cells=-1, persistent=persistent,
                    **kw) as s:
            s.set_beta(beta)
            phi, st = s.solve(f, tol=1e-10)
            assert st["status"] == "ok"
            out.append(phi.cpu().numpy())
    ref, _ = O.solve(d["beta"], d["f"], d["dx"], tol=1e-13)
    assert np.linalg.norm(out[0] - out[1]) <= 1e-12 * np.linalg.norm(ref)
    assert np.linalg.norm(out[0] - ref) <= 1e-9 * np.linalg.norm(ref)


def test_folded_red_pass_on_a_coupled_level(cuda_device):
    # 8 boxes of 48^3 as one 96^3 domain against the single box
    n, m = 96, 48
    d = inputs.stellar(n, 29)
    los = [(i * m, j * m, k * m) for k in (0, 1) for j in (0, 1) for i in (0, 1)]
    cut = lambda a: [a[k:k + m, j:j + m, i:i + m] for i, j, k in los]  # noqa: E731
    s = LevelSolver(los, [(m, m, m)] * 8, d["dx"], device=cuda_device)
    s.set_beta(s.pack([torch.from_numpy(np.ascontiguousarray(b)) for b in cut(d["beta"])]).to(cuda_device))
    phi, st = s.solve(s.pack([torch.from_numpy(np.ascontiguousarray(b))
                              for b in cut(d["f"])]).to(cuda_device), tol=1e-10)
    assert st["status"] == "ok"
    got = np.zeros((n, n, n))
    for q, a in zip(cut(got), s.unpack(phi.cpu())):
        q[...] = a.numpy()
    s.close()
    ref, _ = O.solve(d["beta"], d["f"], d["dx"], tol=1e-13)
    assert np.linalg.norm(got - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", ["nan", "inf", "stall", "zero", "tiny"])
def test_fused_norm_and_decision_match_the_host_loop(cuda_device, kind):
    # a single box's device loop forms the norm and decides in one launch; the
    # host-judged loop in two.  Both add the same partials in the same order, so
    # every outcome and the history agree bit for bit.
    shape = (16, 16, 16) if kind == "tiny" else (40, 48, 72)
    nz, ny, nx = shape
    d = inputs.stellar((nx, ny, nz), 35)
    f = np.array(d["f"])
    if kind in ("nan", "inf"):
        f[nz // 2, 3, 5] = np.nan if kind == "nan" else np.inf
    if kind == "zero":
        f[:] = 0.0
    out = []
    for prof in (False, True):
        with Solver(shape, d["dx"], device=cuda_device) as s:
            s.profile(prof)
            s.set_beta(torch.from_numpy(np.array(d["beta"])).to(cuda_device))
            try:
                phi, st = s.solve(torch.from_numpy(f).to(cuda_device),
                                  tol=1e-30 if kind == "stall" else 1e-10)
            except MGError as e:   # (a non-finite right-hand side is an error)
                assert kind in ("nan", "inf")
                out.append((np.zeros(1), dict(status=e.name, cycles=0, hist=[])))
                continue
            out.append((phi.cpu().numpy(), st))
    (a, sa), (b, sb) = out
    assert np.array_equal(a, b, equal_nan=True)
    assert sa["status"] == sb["status"] and sa["cycles"] == sb["cycles"]
    assert np.array_equal(sa["hist"], sb["hist"], equal_nan=True)
