"""New parameters after a solve whose cycle was captured: the next solve is that of a
solver made with them, bit for bit (the same launches on the same values)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import RsfdeError, Solver, workloads  # noqa: E402

FORMS = {
    "fp64": dict(),
    "mixed": dict(precond="bf16x3", matvec="fp32", basis="fp64", resid="exact"),
    "fp32": dict(precond="fp32", matvec="fp32", basis="fp64", resid="exact"),
    "df32": dict(precond="fp32", matvec="df32", basis="df32", resid="fp64"),
    "paper": dict(variant="gmres_left", tol=1e-8),
}


def solver(w, **kw):
    return Solver(w["n1"], w["n2"], w["box"], w["in_omega"], w["alpha1"], w["alpha2"], w["kx"], w["ky"], w["dt"],
                  w["eta"], **kw)


# dt moves dt/eta; kx and ky move the powers of two that scale the exact products
@pytest.mark.parametrize("kx,ky,dt", [(1.0, 1.0, 7.0), (40.0, 0.02, 1.0), (0.3, 5.0, 0.2)])
@pytest.mark.parametrize("form", list(FORMS))
def test_solve_after_new_parameters(form, kx, ky, dt):
    w = dict(workloads.random_problem(90, 75, 52), eta=1e-4)
    b = torch.as_tensor(w["field"]).cuda()
    new = dict(w, kx=kx * w["kx"], ky=ky * w["ky"], dt=dt * w["dt"])
    s, fresh = solver(w, **FORMS[form]), solver(new, **FORMS[form])
    s.solve(b)
    s.set_params(new["kx"], new["ky"], new["dt"])
    (x, st), (ref, st_ref) = s.solve(b), fresh.solve(b)
    assert torch.equal(x, ref) and st["iters"] == st_ref["iters"]
    s.close()
    fresh.close()


@pytest.mark.parametrize("form", ["fp64", "mixed"])
def test_a_new_wait_bound_holds_in_a_captured_solve(form):
    w = dict(workloads.random_problem(91, 150, 90), eta=1e-4)
    b = torch.as_tensor(w["field"]).cuda()
    s = solver(w, **FORMS[form])
    x = s.solve(b)[0].clone()
    s.set_wait_cycles(1)
    with pytest.raises(RsfdeError) as e:
        s.solve(b)
    assert e.value.name == "ETIMEOUT"
    s.set_wait_cycles(0)
    assert torch.equal(s.solve(b)[0], x)
    s.close()


def test_changing_the_preconditioner_and_back_rebuilds_what_was_captured():
    w = dict(workloads.random_problem(92, 150, 90), eta=1e-4)
    b = torch.as_tensor(w["field"]).cuda()
    s = solver(w, **FORMS["mixed"])
    x = s.solve(b)[0].clone()
    s.set_options(precond="bf16")  # frees the split-BF16 plan
    held = torch.empty(1 << 26, dtype=torch.uint8, device="cuda")
    s.set_options(precond="bf16x3")
    assert torch.equal(s.solve(b)[0], x)
    del held
    s.close()
