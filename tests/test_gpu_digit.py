"""The FP64 sine transforms, preconditioner and operator as digit products on the tensor
cores, at the edges of their tiles (16, 32, 64 columns, 128 rows, 64-wide K
slices) and up to the largest side they take, against dense extended-precision
products.

Tolerances (relative, 2-norm).  Each product rounds its operand to 55 bits of
the row's largest entry (at most 2^-55 of the row's norm) and its result to
one unit of W; W has at least 50 bits where the operand's row has its largest
entry (n = 1), so 2^-51 at most; the sine matrix is within 2^-55.  Two products: below
4 * 2^-51 = 1.8e-15.  The preconditioner: four products, 8 * 2^-51, the
reciprocal and its product, 2 * 2^-53, and the rounded denominators, 2 * 2^-53:
4.0e-15.  The operator: the middle diagonals in FP64 (six roundings of at most
2^-53 of the coefficients' sum times the largest norm they meet) and two products
of the rest, whose coefficients are at most 1/48 of that sum: 8 * 2^-53."""
import numpy as np
import pytest

from paper_2102_11576_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import RsfdeError, Solver  # noqa: E402

SIZES = [(1, 1), (2, 3), (15, 17), (31, 33), (63, 32), (64, 65), (127, 129), (128, 16), (130, 257), (9, 513),
         (2047, 5), (5, 2048)]


def solver(w, **kw):
    return Solver(w["n1"], w["n2"], w["box"], w["in_omega"], w["alpha1"], w["alpha2"], w["kx"], w["ky"], w["dt"],
                  w["eta"], **kw)


def sine(n):
    m = np.arange(2 * (n + 1), dtype=np.longdouble)
    t = np.sqrt(np.longdouble(2) / (n + 1)) * np.sin(np.longdouble("3.14159265358979323846264338327950288") * m / (n + 1))
    i = np.arange(1, n + 1)
    return t[(i[:, None] * i[None, :]) % (2 * (n + 1))]


def off(got, ref):
    return float(np.sqrt(((got - ref) ** 2).sum() / (ref ** 2).sum()))


@pytest.mark.parametrize("n1,n2", SIZES)
def test_products_at_tile_edges(n1, n2):
    w = workloads.random_problem(40, n1, n2)
    s = solver(w)
    v = torch.as_tensor(w["field"]).cuda()
    Sx, Sy, x = sine(n1), sine(n2), w["field"].astype(np.longdouble)
    W = Sy @ x @ Sx
    assert off(s.dst2(v).cpu().numpy(), W) <= 1.8e-15
    t, pen = s.tables(), np.longdouble(s.params()["pen"])
    base = 1 - t["lam_x"].astype(np.longdouble)[None, :] - t["lam_y"].astype(np.longdouble)[:, None]
    z = s.apply_precond(v).cpu().numpy()
    for out, den in ((False, base), (True, base + pen)):
        ref, sel = Sy @ (W / den) @ Sx, (w["in_omega"] == 0) == out
        if sel.any():  # each channel against its own scale (the penalised one is far smaller)
            assert np.abs(z - ref)[sel].max() <= 4.0e-15 * np.sqrt((ref ** 2).sum())
    s.close()


@pytest.mark.parametrize("n1,n2", SIZES)
def test_operator_at_tile_edges(n1, n2):
    w = workloads.random_problem(43, n1, n2)
    s = solver(w)
    v = torch.as_tensor(w["field"]).cuda()
    t, pen, z = s.tables(), np.longdouble(s.params()["pen"]), w["field"].astype(np.longdouble)
    Tx, Ty = (t[k].astype(np.longdouble)[np.abs(np.subtract.outer(np.arange(n), np.arange(n)))]
              for k, n in (("t_x", n1), ("t_y", n2)))
    out = w["in_omega"] == 0
    ref = z - z @ Tx - Ty @ z + pen * out * z
    err = s.apply_M(v).cpu().numpy() - ref
    scale = 1 + 2 * (np.abs(t["t_x"]).sum() + np.abs(t["t_y"]).sum())
    norm = np.sqrt((z ** 2).sum())
    assert np.sqrt((err[~out] ** 2).sum()) <= 8 * 2.0 ** -53 * scale * norm
    assert np.sqrt((err[out] ** 2).sum()) <= 8 * 2.0 ** -53 * (scale + float(pen)) * norm
    assert torch.equal(s.apply_M(v * 2.0 ** 40), s.apply_M(v) * 2.0 ** 40)
    v[n2 // 2, n1 // 2] = float("nan")
    assert s.apply_M(v).isnan()[n2 // 2].all()
    s.close()


def test_operator_follows_new_parameters_in_a_captured_solve():
    w = workloads.random_problem(44, 75, 52)
    s = solver(w)
    b = torch.as_tensor(w["field"]).cuda()
    s.solve(b)
    s.set_params(40.0 * w["kx"], 0.02 * w["ky"], w["dt"])
    fresh = solver(dict(w, kx=40.0 * w["kx"], ky=0.02 * w["ky"]))
    assert torch.equal(s.apply_M(b), fresh.apply_M(b))
    assert torch.equal(s.solve(b)[0], fresh.solve(b)[0])
    s.close()
    fresh.close()


def test_scaling_zeros_and_non_finite_entries():
    w = workloads.random_problem(41, 70, 45)
    s = solver(w)
    v = torch.as_tensor(w["field"]).cuda()
    v[7] = 0.0
    v[:, 11] = 0.0
    v[20] *= 2.0 ** -80
    z = s.apply_precond(v).clone()
    for k in (-300, 300):  # a power of two passes through exactly
        assert torch.equal(s.apply_precond(v * 2.0 ** k), z * 2.0 ** k)
    assert not s.apply_precond(torch.zeros_like(v)).any()
    for bad in (float("nan"), float("inf")):
        b = v.clone()
        b[3, 5] = bad
        assert s.apply_precond(b).isnan().all() and s.dst2(b).isnan().all()
    assert torch.equal(s.apply_precond(v), z)
    s.close()


def test_a_wait_that_gives_up_is_seen_and_left_behind():
    w = workloads.random_problem(42, 150, 90)
    s = solver(w, use_graph=False)
    v = torch.as_tensor(w["field"]).cuda()
    z = s.apply_precond(v).clone()
    s.set_wait_cycles(1)  # every pipeline wait that is not already satisfied gives up
    assert s.apply_precond(v).isnan().any()
    with pytest.raises(RsfdeError) as e:
        s.solve(v)
    assert e.value.name == "ETIMEOUT"
    s.set_wait_cycles(0)
    assert torch.equal(s.apply_precond(v), z)
    x, st = s.solve(v)
    assert st["converged"] and (s.residual(x, v).norm() <= 1.01e-10 * v.norm()).item()
    s.close()
