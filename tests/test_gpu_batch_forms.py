"""The batch on forms and sizes that test_gpu_batch.py does not reach."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import Batch, RsfdeError, Solver, workloads  # noqa: E402


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


# FP64: every instance a branch of the graph, with digit products; bf16x3: grouped GEMMs in lock step;
# the other two as branches again, with GEMMs of their own (and FP64 digit products beside them)
TIMED = [dict(precond="fp64", matvec="fp64", basis="fp64", resid="fp64"),
         dict(precond="bf16x3", matvec="fp32", basis="fp64", resid="exact"),
         dict(precond="bf16x3", matvec="df32", basis="df32", resid="fp64"),
         dict(precond="bf16x3", matvec="fp64", basis="fp64", resid="fp64")]


@pytest.mark.parametrize("form", TIMED)
def test_a_wait_that_gives_up_fails_the_run_and_is_left_behind(form):
    ws = problems([(75, 52), (40, 33), (150, 90)])
    b = Batch(ws, **form)

    def march():
        for i, w in enumerate(ws):
            b.set(i, w["field"])
        b.run(2)
        return [b.get(i) for i in range(len(ws))]

    ref = march()
    b.set_wait_cycles(1)  # every pipeline wait that is not already satisfied gives up
    with pytest.raises(RsfdeError) as e:
        march()
    assert e.value.name == "ETIMEOUT"
    b.set_wait_cycles(0)
    for got, want in zip(march(), ref):
        assert torch.equal(got, want)
    b.close()


@pytest.mark.parametrize("form", TIMED)
def test_a_solve_reports_its_own_give_ups_only(form):
    w, = problems([(150, 90)])
    v = torch.as_tensor(w["field"]).cuda()
    s = single(w, **form)
    x = s.solve(v)[0].clone()
    s.set_wait_cycles(1)
    with pytest.raises(RsfdeError) as e:
        s.solve(v)
    assert e.value.name == "ETIMEOUT"
    if form["matvec"] == "fp64":
        assert s.apply_M(v).isnan().any()
    if form["precond"] == "fp64":
        assert s.apply_precond(v).isnan().any() and s.dst2(v).isnan().any()
    s.set_wait_cycles(0)
    assert torch.equal(s.solve(v)[0], x)
    s.close()
