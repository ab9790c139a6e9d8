"""The work that users of this framework have it do, as cases to be timed.

A case is a plain dict; ``prepare`` makes the fields on the GPU and the solver
that a program keeps, ``run`` is one pass through the public entry points,
``work`` says what that pass cannot do without, and ``exact`` gives its result
in 64 bits by dense torch algebra written from the formulas of the method
(Eq. 2.17, Eq. 4.6), without this package.

Kinds (``case["kind"]``):
  step      one implicit time step, the call a time march repeats (Solver.step)
  paper     one solve in the paper's own mode, left-preconditioned GMRES(20) to
            1e-8 (Solver.solve with variant="gmres_left")
  batch     one step of many small independent problems (Batch.set/run/get)
  gradient  a short differentiable march and its backward pass (adjoint.march)
  apply_M, precond, residual, dst2
            the single operators that a program composes its own solver from
Forms (``case["form"]``): "fp64" is the library's default, "mixed" the split
BF16 / FP32 / exact-residual form that the benchmark leads with, "fp32" the
FP32 preconditioner beside the same FP64 basis (with the exact residual).
"""
import math

import numpy as np
import torch

from paper_2102_11576_gb300 import Batch, Solver
from paper_2102_11576_gb300.adjoint import march

BOX = (-1.0, 1.0, -1.0, 1.0)
ETA = 1e-8
FORMS = {
    "fp64": dict(precond="fp64", matvec="fp64", basis="fp64", resid="fp64"),
    "mixed": dict(precond="bf16x3", matvec="fp32", basis="fp64", resid="exact"),
    "fp32": dict(precond="fp32", matvec="fp32", basis="fp64", resid="exact"),
}
DOMAINS = ("disk", "ellipse", "polygon")


def listed():
    def case(name, kind, form, n1, n2, **kw):
        return dict(dict(name=name, kind=kind, form=form, n1=n1, n2=n2, a1=1.5, a2=1.7, kx=1.0, ky=1.0, dt=0.02,
                         domain="disk", restart=20), **kw)

    return [
        # the benchmark's smallest march: a 64 x 64 disk in the default FP64 form (launch and latency bound)
        case("step_fp64_64", "step", "fp64", 64, 64, dt=1.0 / 64),
        # its medium march: 512 x 512 ellipse with a source, FGMRES(30), FP64
        case("step_fp64_512", "step", "fp64", 512, 512, a1=1.2, a2=1.8, kx=2.0, ky=0.5, dt=0.01, domain="ellipse",
             restart=30),
        # the headline workload in the default FP64 form: the largest call here
        case("step_fp64_2048", "step", "fp64", 2048, 2048, a1=1.3, a2=1.6, domain="polygon"),
        # the headline workload in the headline form
        case("step_mixed_2048", "step", "mixed", 2048, 2048, a1=1.3, a2=1.6, domain="polygon"),
        # the headline form on a grid that nothing was tuned for: odd sides, two transform lengths
        case("step_mixed_1201x777", "step", "mixed", 1201, 777, a1=1.4, a2=1.55, kx=0.8, ky=1.6, domain="ellipse"),
        # parameter studies: many small problems of uneven size at once
        case("batch_mixed_48", "batch", "mixed", 64, 512, count=48, dt=0.05),
        # fitting k and a source to data: forward and backward of a short march
        case("gradient_mixed_512", "gradient", "mixed", 512, 512, a1=1.5, a2=1.5, dt=0.01, steps=3),
        # a row of the paper's Table 1 (n = 128, one of its 128 steps)
        case("paper_fp64_128", "paper", "fp64", 128, 128, a1=1.4, a2=1.7, dt=1.0 / 128),
        # the operators for a caller's own Krylov method, FP64, odd and ragged sides
        case("precond_fp64_1023x641", "precond", "fp64", 1023, 641),
        case("apply_M_fp64_300x1500", "apply_M", "fp64", 300, 1500, a1=1.25, a2=1.85),
        # the true residual that decides convergence, at the headline size
        case("residual_exact_2048", "residual", "mixed", 2048, 2048, a1=1.3, a2=1.6, domain="polygon"),
        # a small sine transform (spectral filtering of one field)
        case("dst2_fp64_96x200", "dst2", "fp64", 96, 200),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "step", "batch", "gradient", "paper", "precond", "apply_M", "residual", "dst2"))
    c = dict(kind=kind, form="fp64", a1=round(rng.uniform(1.1, 1.9), 3), a2=round(rng.uniform(1.1, 1.9), 3),
             kx=round(rng.uniform(0.5, 2.0), 3), ky=round(rng.uniform(0.5, 2.0), 3),
             dt=round(rng.uniform(0.005, 0.03), 4), domain=rng.choice(DOMAINS), restart=rng.choice((20, 20, 30)))
    if kind == "batch":
        lo = logint(16, 100)
        c.update(form=rng.choice(("mixed", "mixed", "fp32")), n1=lo, n2=min(512, logint(2 * lo, 8 * lo)),
                 count=logint(4, 48), restart=20, dt=0.05)
        return c
    if kind in ("step", "gradient", "paper"):
        top = {"step": 2048, "gradient": 512, "paper": 512}[kind]
        c["n1"] = logint(32, top)
        c["n2"] = min(top, max(32, int(c["n1"] * 2.0 ** rng.uniform(-1.0, 1.0))))
        if kind != "paper":
            c["form"] = rng.choice(("fp64", "mixed", "mixed", "fp32"))
        if kind == "step" and c["form"] == "fp64":  # about the time of the largest listed call at most
            while c["n1"] * c["n2"] > 1500 * 1500:
                c["n1"], c["n2"] = c["n1"] * 3 // 4, c["n2"] * 3 // 4
        if kind == "gradient":
            c.update(steps=rng.choice((2, 3)), restart=20)
        if kind == "paper":
            c.update(restart=20)
        return c
    while True:  # single operators: any two sides the library takes, up to the headline's cell count
        c["n1"], c["n2"] = logint(24, 4096), logint(24, 4096)
        if c["n1"] * c["n2"] <= 2048 * 2048:
            break
    c["form"] = "mixed" if kind == "residual" else "fp64"
    return c


# ---- inputs --------------------------------------------------------------------
def _fields(case, seed, n1, n2, device, domain):
    """A domain mask and smooth fields on it: the mid-march pair u^{k-1}, u^{k-2} and a source."""
    r = np.random.default_rng(seed)
    x = torch.linspace(-1.0, 1.0, n1 + 2, dtype=torch.float64, device=device)[1:-1][None, :]
    y = torch.linspace(-1.0, 1.0, n2 + 2, dtype=torch.float64, device=device)[1:-1][:, None]
    if domain == "disk":
        s = r.uniform(0.9, 1.0)
        q = (x / s) ** 2 + (y / s) ** 2
        inside = q <= 1.0
    elif domain == "ellipse":
        a, b, th = r.uniform(0.75, 0.95), r.uniform(0.55, 0.9), r.uniform(0.0, math.pi)
        xr, yr = math.cos(th) * x + math.sin(th) * y, -math.sin(th) * x + math.cos(th) * y
        q = (xr / a) ** 2 + (yr / b) ** 2
        inside = q <= 1.0
    else:  # a convex polygon around the centre, its vertices near the unit circle
        k = int(r.integers(8, 13))
        ang = (np.arange(k) + r.uniform(0.1, 0.9, size=k)) * (2.0 * math.pi / k)
        inside = torch.ones((n2, n1), dtype=torch.bool, device=device)
        for e in range(k):
            x0, y0, x1, y1 = (float(f(ang[(e + d) % k])) for d in (0, 1) for f in (np.cos, np.sin))
            inside &= (x1 - x0) * (y - y0) - (y1 - y0) * (x - x0) >= 0.0
        q = x ** 2 + y ** 2
    u = torch.clamp(1.0 - q, min=0.0) ** 2

    def bumps(count, amp):
        f = torch.zeros((n2, n1), dtype=torch.float64, device=device)
        for _ in range(count):
            x0, y0 = r.uniform(-0.5, 0.5, size=2)
            f += r.uniform(-amp, amp) * torch.exp(-((x - x0) ** 2 + (y - y0) ** 2) / (2.0 * r.uniform(0.1, 0.3) ** 2))
        return f

    u = u * (1.0 + bumps(3, 0.3)) * inside
    older = u * (1.0 + case["dt"] * bumps(3, 2.0))
    return inside, u.contiguous(), older.contiguous(), bumps(2, 1.0).contiguous()


def _problem(case, seed, device):
    inside, u, older, src = _fields(case, seed, case["n1"], case["n2"], device, case["domain"])
    return dict(n1=case["n1"], n2=case["n2"], a1=case["a1"], a2=case["a2"], kx=case["kx"], ky=case["ky"],
                dt=case["dt"], inside=inside, u=u, older=older, src=src)


def _batch_problems(case, seed, device):
    """case["count"] problems of their own size, domain and parameters (those of make_batch)."""
    r = np.random.default_rng(seed)
    out = []
    sizes = np.linspace(case["n1"], case["n2"], case["count"]).astype(int)  # the same sizes for every seed
    for i, n in enumerate(sizes):
        n = int(n) + (i % 2 if n < case["n2"] else 0)
        inside, u, older, src = _fields(case, int(r.integers(1 << 30)), n, n, device,
                                        DOMAINS[1 + int(r.integers(2))])
        out.append(dict(n1=n, n2=n, a1=float(r.uniform(1.1, 1.9)), a2=float(r.uniform(1.1, 1.9)),
                        kx=float(r.uniform(0.5, 2.0)), ky=float(r.uniform(0.5, 2.0)), dt=case["dt"], inside=inside,
                        u=u, older=older, src=src))
    return out


def _inputs(case, seed, device):
    """The operators' operand: a smooth field with noise, as a Krylov vector has."""
    p = _problem(case, seed, device)
    g = torch.Generator(device=device).manual_seed(seed)
    noise = torch.randn((case["n2"], case["n1"]), generator=g, dtype=torch.float64, device=device)
    p["v"] = (p["u"] + 0.1 * noise * p["inside"]).contiguous()
    return p


def _solver(p, case, **kw):
    return Solver(p["n1"], p["n2"], BOX, p["inside"], p["a1"], p["a2"], p["kx"], p["ky"], p["dt"], ETA,
                  restart=case["restart"], **FORMS[case["form"]], **kw)


def prepare(case, seed):
    device, kind = torch.device("cuda"), case["kind"]
    if kind == "batch":
        ps = _batch_problems(case, seed, device)
        b = Batch([dict(n1=p["n1"], n2=p["n2"], box=BOX, in_omega=p["inside"].cpu().numpy(), alpha1=p["a1"],
                        alpha2=p["a2"], kx=p["kx"], ky=p["ky"], dt=p["dt"], eta=ETA) for p in ps],
                  restart=case["restart"], **FORMS[case["form"]])
        return dict(kind=kind, batch=b, ps=ps)
    if kind in ("step", "gradient", "paper"):
        p = _problem(case, seed, device)
    else:
        p = _inputs(case, seed, device)
    if kind == "paper":
        s = _solver(p, case, tol=1e-8, variant="gmres_left")
        b = p["u"] + p["dt"] * p["src"] * p["inside"]
        return dict(kind=kind, solver=s, p=p, b=b, guess=2.0 * p["u"] - p["older"])
    s = _solver(p, case, tol=1e-12) if kind == "gradient" else _solver(p, case)
    if kind == "gradient":
        p["target"] = (0.5 * p["u"]).contiguous()
        p["leaves"] = [p["u"].clone().requires_grad_(True), torch.tensor(p["kx"], dtype=torch.float64,
                                                                          requires_grad=True),
                       torch.tensor(p["ky"], dtype=torch.float64, requires_grad=True),
                       p["src"].clone().requires_grad_(True)]
        p["steps"] = case["steps"]
    return dict(kind=kind, solver=s, p=p, out=s.empty())


def run(state):
    kind = state["kind"]
    if kind == "batch":
        b = state["batch"]
        for i, p in enumerate(state["ps"]):
            b.set(i, p["u"], p["src"])
        b.run(1)
        return [b.get(i) for i in range(b.count)]
    s, p = state["solver"], state["p"]
    if kind == "step":
        return s.step(p["u"], p["older"], p["src"], out=state["out"])[0]
    if kind == "paper":
        return s.solve(state["b"], state["guess"].clone())[0]
    if kind == "gradient":
        u0, kx, ky, src = p["leaves"]
        u = march(s, u0, kx, ky, src, steps=p["steps"])
        loss = ((u - p["target"]) ** 2).sum()
        return [u.detach()] + list(torch.autograd.grad(loss, [u0, kx, ky, src]))
    if kind == "apply_M":
        return s.apply_M(p["v"], out=state["out"])
    if kind == "precond":
        return s.apply_precond(p["v"], out=state["out"])
    if kind == "residual":
        return s.residual(p["v"], p["u"], out=state["out"])
    return s.dst2(p["v"], out=state["out"])


# ---- what a pass cannot do without --------------------------------------------
def _transform_flops(n1, n2):
    """One real transform (or Toeplitz product) of every row and every column by FFT."""
    return sum(m * 2.5 * 2 * n * math.log2(2 * n) * 2 for n, m in ((n1, n2), (n2, n1)))


def _solve_work(n1, n2, iters, form, restart):
    """A Krylov solve of `iters` iterations: per iteration the operator, the three sine-transform pairs of the
    preconditioner, and the dots and updates against the basis (each basis vector read once)."""
    N, ez = n1 * n2, 8.0 if form == "fp64" else 4.0
    cycles = max(1.0, iters / restart)
    mean_j = min(iters, restart) / 2.0
    per_it = N * (2.0 * (8.0 + ez) + 8.0 * (mean_j + 2.0))
    flops = iters * (_transform_flops(n1, n2) * 4.0 + 4.0 * N * (mean_j + 1.0))
    return per_it * iters + cycles * N * 40.0, flops + cycles * _transform_flops(n1, n2)


def work(case):
    kind, n1, n2 = case["kind"], case["n1"], case["n2"]
    N = n1 * n2
    if kind == "batch":
        sizes = np.linspace(n1, n2, case["count"])
        parts = [_solve_work(n, n, max(12.0, 8.0 * math.log2(n) - 32.0), case["form"], 20) for n in sizes]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind in ("step", "gradient", "paper"):
        iters = max(12.0, 4.0 * math.log2(N) - 32.0) if kind != "paper" else 5.0
        b, f = _solve_work(n1, n2, iters, case["form"], case["restart"])
        k = 2 * case["steps"] if kind == "gradient" else 1
        return {"bytes": k * b, "flops": k * f}
    t = _transform_flops(n1, n2)
    return {"bytes": {"residual": 25.0, "precond": 17.0, "apply_M": 17.0, "dst2": 16.0}[kind] * N,
            "flops": {"residual": t, "apply_M": t, "dst2": t, "precond": 3.0 * t}[kind]}


# ---- the same in 64 bits -----------------------------------------------------
class _Dense:
    """M and P-hat^-1 of one problem as dense FP64 matrices per axis."""

    def __init__(self, p, device):
        def axis(n, alpha, k):
            h = 2.0 / (n + 1)
            c = p["dt"] * k * (-1.0 / (2.0 * math.cos(alpha * math.pi / 2.0))) / h ** alpha
            g = np.cumprod(np.concatenate([[1.0], 1.0 - (alpha + 1.0) / np.arange(1, n + 2)]))
            t = c * np.concatenate([[2.0 * g[1]], [g[0] + g[2]], g[3:n + 1]])[:n]
            d = torch.as_tensor(t, device=device)
            i = torch.arange(n, device=device)
            T = d[(i[:, None] - i[None, :]).abs()]
            j = torch.arange(1, n + 1, device=device)
            ph = (j[:, None] * j[None, :]) % (2 * (n + 1))
            S = math.sqrt(2.0 / (n + 1)) * torch.sin(math.pi * ph.double() / (n + 1))
            lam = d[0] + 2.0 * torch.cos(math.pi * ph.double() / (n + 1))[:, :n - 1] @ d[1:]
            return T, S, lam

        self.Tx, self.Sx, lx = axis(p["n1"], p["a1"], p["kx"])
        self.Ty, self.Sy, ly = axis(p["n2"], p["a2"], p["ky"])
        self.pen = p["dt"] / ETA
        self.out = ~p["inside"]
        self.base = 1.0 - lx[None, :] - ly[:, None]

    def M(self, z):
        return z - z @ self.Tx - self.Ty @ z + self.pen * self.out * z

    def dst2(self, v):
        return self.Sy @ v @ self.Sx

    def P(self, v):
        w = self.dst2(v)
        return torch.where(self.out, self.dst2(w / (self.base + self.pen)), self.dst2(w / self.base))

    def solve(self, b, x=None, tol=2e-14):
        """M x = b by right-preconditioned GMRES with re-orthogonalisation, restarted on the true residual."""
        x = torch.zeros_like(b) if x is None else x
        bn = b.norm()
        last = math.inf
        for _ in range(4):
            r = b - self.M(x)
            beta = float(r.norm())
            if beta <= tol * bn or beta > 0.3 * last:
                break
            last = beta
            m = min(150, b.numel())
            V = torch.zeros((m + 1, b.numel()), dtype=b.dtype, device=b.device)
            Z, H = [], np.zeros((m + 1, m))
            V[0] = r.flatten() / beta
            for j in range(m):
                Z.append(self.P(V[j].view_as(b)))
                w = self.M(Z[j]).flatten()
                h = V[:j + 1] @ w
                w = w - h @ V[:j + 1]
                h2 = V[:j + 1] @ w
                w = w - h2 @ V[:j + 1]
                nw = float(w.norm())
                H[:j + 1, j], H[j + 1, j] = (h + h2).cpu().numpy(), nw
                e = np.zeros(j + 2)
                e[0] = beta
                y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) <= max(1e-8 * beta, 0.3 * tol * float(bn)) or nw == 0.0:
                    break
                V[j + 1] = w / nw
            for c, z in zip(y, Z):
                x = x + float(c) * z
        return x

    def step(self, u, src, dt, guess):
        return self.solve(u + dt * torch.where(self.out, 0.0, u - u ** 3 + src), guess)


def exact(case, seed):
    device, kind = torch.device("cuda"), case["kind"]
    if kind == "batch":
        outs = []
        for p in _batch_problems(case, seed, device):
            outs.append(_Dense(p, device).step(p["u"], p["src"], p["dt"], p["u"]))
        return outs
    if kind in ("step", "paper", "gradient"):
        p = _problem(case, seed, device)
        d = _Dense(p, device)
        if kind == "step":
            return d.step(p["u"], p["src"], p["dt"], p["u"])
        if kind == "paper":
            return d.solve(p["u"] + p["dt"] * p["src"] * p["inside"], p["u"])
        us, tgt = [p["u"]], 0.5 * p["u"]
        for _ in range(case["steps"]):
            us.append(d.step(us[-1], p["src"], p["dt"], us[-1]))
        lam, gs = 2.0 * (us[-1] - tgt), torch.zeros_like(tgt)
        gx = gy = 0.0
        for k in range(case["steps"], 0, -1):
            mu = d.solve(lam, lam)
            gx += float((mu * (us[k] @ d.Tx)).sum()) / p["kx"]
            gy += float((mu * (d.Ty @ us[k])).sum()) / p["ky"]
            inner = torch.where(d.out, 0.0, p["dt"] * mu)
            gs += inner
            lam = mu + inner * (1.0 - 3.0 * us[k - 1] ** 2)
        return [us[-1], lam, torch.tensor(gx, dtype=torch.float64), torch.tensor(gy, dtype=torch.float64), gs]
    p = _inputs(case, seed, device)
    d = _Dense(p, device)
    if kind == "apply_M":
        return d.M(p["v"])
    if kind == "precond":
        return d.P(p["v"])
    if kind == "residual":
        return p["u"] - d.M(p["v"])
    return d.dst2(p["v"])
