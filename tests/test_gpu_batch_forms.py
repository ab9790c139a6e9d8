"""The batch on forms and sizes that test_gpu_batch.py does not reach."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import Batch, Solver, workloads  # noqa: E402


def problems(sizes):
    ws = [dict(workloads.random_problem(80 + i, n1, n2), eta=1e-4) for i, (n1, n2) in enumerate(sizes)]
    for w in ws:
        w["field"] = np.abs(w["field"]) * 0.1 * w["in_omega"]
    return ws


def single(w, **form):
    return Solver(w["n1"], w["n2"], w["box"], w["in_omega"], w["alpha1"], w["alpha2"], w["kx"], w["ky"], w["dt"],
                  w["eta"], **form)


# sides up to 8 take transforms of length 16, whose groups fill the most shared memory
@pytest.mark.parametrize("form", [dict(precond="bf16x3", matvec="fp32", basis="fp64", resid="exact"),
                                  dict(precond="fp32", matvec="fp32", basis="fp64", resid="exact"),
                                  dict(precond="fp32", matvec="fp32", basis="fp64", resid="fp64")])
def test_short_sides_equal_single_solves(form):
    ws = problems([(17, 3), (8, 40), (5, 7), (1, 9), (9, 9)])
    b = Batch(ws, **form)
    for i, w in enumerate(ws):
        b.set(i, w["field"])
    b.run(1)
    for i, w in enumerate(ws):
        s = single(w, **form)
        assert torch.equal(b.get(i), s.step(torch.as_tensor(w["field"]).cuda())[0])
        s.close()
    b.close()
