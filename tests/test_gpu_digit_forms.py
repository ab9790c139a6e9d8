"""The FP64 forms' digit products on what test_gpu_digit.py does not reach."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_11576_gb300 import workloads  # noqa: E402
from test_gpu_digit import off, sine, solver  # noqa: E402


def few_rows(w, count=8):
    """A field that is zero but for `count` rows, the first and the last among them, and those rows."""
    rows = np.unique(np.linspace(0, w["n2"] - 1, count).astype(int))
    z = np.zeros_like(w["field"])
    z[rows] = w["field"][rows]
    return z, rows


def operator_error(s, w, got, z, rows):
    """|got - M z| over and outside Omega and its bound there, in units of |z| (2-norm): M's middle
    diagonals in FP64, six roundings of at most 2^-53 of the coefficients' sum, and
    two products of the rest: 8 * 2^-53 of that sum."""
    t, pen = s.tables(), np.longdouble(s.params()["pen"])
    tx, ty = t["t_x"].astype(np.longdouble), t["t_y"].astype(np.longdouble)
    zl, ref, out = z[rows].astype(np.longdouble), z.astype(np.longdouble), w["in_omega"] == 0
    n1, n2 = w["n1"], w["n2"]
    ref[rows] -= zl @ tx[np.abs(np.subtract.outer(np.arange(n1), np.arange(n1)))]
    ref -= ty[np.abs(np.subtract.outer(np.arange(n2), rows))] @ zl
    ref += pen * out * z
    err, norm = got - ref, np.sqrt((z.astype(np.longdouble) ** 2).sum())
    scale = 1 + 2 * (np.abs(tx).sum() + np.abs(ty).sum())
    return [(np.sqrt((err[sel] ** 2).sum()), 8 * 2.0 ** -53 * c * norm) for sel, c in ((~out, scale), (out, scale + pen))]


# four columns of the fold in shared memory: 48 KB, or less by up to the kernel's static 1 KB
@pytest.mark.parametrize("n1,n2", [(608, 1503), (608, 1504), (609, 1535), (608, 1536)])
def test_operator_near_the_plain_limit_of_shared_memory(n1, n2):
    w = workloads.random_problem(70, n1, n2)
    z, rows = few_rows(w)
    s = solver(w)
    for err, bound in operator_error(s, w, s.apply_M(torch.as_tensor(z).cuda()).cpu().numpy(), z, rows):
        assert err <= bound
    s.close()


@pytest.mark.parametrize("n1,n2", [(1, 1), (33, 31), (64, 65), (70, 129)])
def test_operators_in_place(n1, n2):
    w = workloads.random_problem(71, n1, n2)
    s = solver(w)
    v = torch.as_tensor(w["field"]).cuda()
    for op in (s.apply_M, s.apply_precond, s.dst2):
        ref, x = op(v), v.clone()
        assert torch.equal(op(x, out=x), ref)
    s.close()


def test_autotune_still_takes_the_fp64_transforms():
    w = workloads.random_problem(72, 100, 70)
    s = solver(w)
    chosen = s.autotune(reps=1)  # rsfde_residual and the adjoint run them beside the digit products
    assert {"toeplitz_rows", "toeplitz_cols", "dst_rows", "precond_cols", "precond_rows"} <= set(chosen)
    s.close()


def test_sides_without_digit_products_are_tried_once():
    """A try makes three tables of 4,096 long-double sines and waits for three kernels."""
    took = {}
    for n1 in (2047, 2048):  # no scale of S_2047's digits keeps the sums exact
        w = workloads.random_problem(73, n1, 5)
        s = solver(w)
        calls = []
        for _ in range(20):
            t = time.perf_counter()
            s.set_options(tol=1e-10)
            calls.append(time.perf_counter() - t)
        took[n1] = min(calls)
        s.close()
    assert took[2047] <= 5 * took[2048]


def sampled_errors(s, w, z, rows, Sx, Sy):
    """dst2 as a whole, and P-hat^-1 over eight rows and eight columns of either channel, relative to
    the 2-norm of the transform (test_gpu_digit's bounds)."""
    v = torch.as_tensor(z).cuda()
    W = Sy[:, rows] @ (z[rows].astype(np.longdouble) @ Sx)
    yield off(s.dst2(v).cpu().numpy(), W), 1.8e-15
    t, pen = s.tables(), np.longdouble(s.params()["pen"])
    base = 1 - t["lam_x"].astype(np.longdouble)[None, :] - t["lam_y"].astype(np.longdouble)[:, None]
    got = s.apply_precond(v).cpu().numpy()
    ys = np.unique(np.linspace(0, w["n2"] - 1, 8).astype(int))
    xs = np.unique(np.linspace(0, w["n1"] - 1, 8).astype(int))
    for out, den in ((False, base), (True, base + pen)):
        q = W / den
        sel, norm = (w["in_omega"] == 0) == out, np.sqrt((q ** 2).sum())
        for at, ref in ((np.s_[ys, :], (Sy[ys] @ q) @ Sx), (np.s_[:, xs], Sy @ (q @ Sx[:, xs]))):
            if sel[at].any():
                yield np.abs(got[at] - ref)[sel[at]].max() / norm, 4.0e-15


# tiles of 32 and 64 columns, which the smaller sides of test_gpu_digit.py do not take (dg_bn):
# P-hat^-1's four products and the operator's two have the widths
#   1023 x 641: 32 32 64 64, 32 32    257 x 1999: 16 32 16 64, 32 32    2045 x 300: 32 32 64 64, 16 32
#   1101 x 1099: 64 64 32 32, 64 64
@pytest.mark.parametrize("n1,n2", [(1023, 641), (257, 1999), (2045, 300), (1101, 1099)])
def test_wider_tiles(n1, n2):
    w = workloads.random_problem(74, n1, n2)
    z, rows = few_rows(w)
    s = solver(w)
    for err, bound in sampled_errors(s, w, z, rows, sine(n1), sine(n2)):
        assert err <= bound
    for err, bound in operator_error(s, w, s.apply_M(torch.as_tensor(z).cuda()).cpu().numpy(), z, rows):
        assert err <= bound
    s.close()


@pytest.mark.parametrize("n1,n2", [(1023, 641), (1101, 1099)])
def test_a_wait_that_gives_up_on_wider_tiles(n1, n2):
    w = workloads.random_problem(75, n1, n2)
    s = solver(w)
    v = torch.as_tensor(w["field"]).cuda()
    ops = (s.apply_precond, s.dst2, s.apply_M)
    ref = [op(v).clone() for op in ops]
    s.set_wait_cycles(1)  # every pipeline wait that is not already satisfied gives up
    for op in ops:
        assert op(v).isnan().any()
    s.set_wait_cycles(0)
    for op, want in zip(ops, ref):
        assert torch.equal(op(v), want)
    s.close()
