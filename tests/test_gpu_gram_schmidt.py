"""Gram-Schmidt at the edges of its packs (two FP64 or double-FP32 elements, four FP32
ones), of its blocks' shares (1 to 4 packs of 256 threads, up to 64 blocks of one) and on
odd grids, whose last elements are taken one by one and whose packs cross
rows in the BF16 operand.

Tolerance of a solve: M is symmetric with eigenvalues >= 1, so a solution with
||b - M x|| <= tol ||b|| is within tol ||b|| of the exact one; two such solutions
differ by 2 tol ||b|| at most (tol = 1e-10), and the true residuals themselves
are evaluated to below 1e-10 ||b||: 3e-10 ||b||."""
import numpy as np
import pytest

import oracle
from paper_2102_11576_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import Batch, RsfdeError, Solver  # noqa: E402

FORMS = {
    "fp64": dict(),
    "mixed": dict(precond="bf16x3", matvec="fp32", basis="fp64", resid="exact"),
    "df32": dict(precond="fp32", matvec="df32", basis="df32", resid="fp64"),
    "fp32": dict(precond="bf16x3", matvec="fp32", basis="fp32", resid="fp64"),
}
# N = 1, 3 and 5 (less than a pack, a pack and a tail), 511 x 1 (one block's packs), odd x odd,
# odd x even, N mod 4 = 1, 2, 3, and 363 x 181 = 65703: more than 64 blocks of one pack
SIZES = [(1, 1), (3, 1), (1, 5), (511, 1), (33, 31), (31, 34), (64, 65), (129, 127), (363, 181)]


def args(w):
    return (w["n1"], w["n2"], w["box"], w["in_omega"], w["alpha1"], w["alpha2"], w["kx"], w["ky"], w["dt"], w["eta"])


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("n1,n2", SIZES)
def test_solve_on_odd_grids(n1, n2, form):
    w = dict(workloads.random_problem(50, n1, n2), eta=1e-4)
    s = Solver(*args(w), restart=20, tol=1e-10, **FORMS[form])
    b = torch.as_tensor(w["field"]).cuda()
    x, st = s.solve(b)
    ref = oracle.Problem(*args(w)).fgmres(w["field"], tol=1e-10)[0]
    assert st["converged"]
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 3e-10 * np.linalg.norm(w["field"])
    # what a vector holds past its last element is never read: a solve that ends
    # in NaN everywhere leaves nothing behind
    x0 = x.clone()
    bad = b.clone()
    bad[0, 0] = float("nan")
    try:
        s.solve(bad)
    except RsfdeError:
        pass
    assert torch.equal(s.solve(b)[0], x0)
    s.close()


def test_batch_of_odd_grids_equals_single_solves():
    sizes = [(33, 31), (31, 34), (64, 65), (17, 11), (129, 127)]
    ws = [dict(workloads.random_problem(60 + i, n1, n2), eta=1e-4) for i, (n1, n2) in enumerate(sizes)]
    for w in ws:
        w["field"] = np.abs(w["field"]) * 0.1 * w["in_omega"]
    b = Batch(ws, **FORMS["mixed"])
    for i, w in enumerate(ws):
        b.set(i, w["field"])
    b.run(1)
    for i, w in enumerate(ws):
        s = Solver(*args(w), **FORMS["mixed"])
        assert torch.equal(b.get(i), s.step(torch.as_tensor(w["field"]).cuda())[0])
        s.close()
    b.close()
