"""Performance cases: whole calls of the library as its users make them.

A time-stepping case ("fs": the semi-implicit Fourier-spectral scheme, "fd": the explicit finite-difference one, in 2D and
3D) sets the fields of a plan from device memory, advances it and reads the fields back.  "ensemble" does the same for many
2D simulations of uneven size in one plan, "trajectory" runs the differentiable trajectory forward and backward, "adjoint"
one adjoint step of a plan.  Each case names its grid (nx, ny, nz; nz = 1 in 2D), the order parameters p, the precision, the
Laplacian (0 spectral, 1 and 2 the finite-difference forms) and the time steps of one pass.
"""
import math

import torch

from paper_2306_04322_gb300 import adjoint, fs
from paper_2306_04322_gb300 import inputs as I


def listed():
    return [
        # a student-size run to its end: 64^2, one order parameter, double precision, 200 steps at five times the FD step
        _case("fs", (64, 64), 1, "f64", 200, start="noise", name="fs2d_64_p1_f64"),
        # one step inside a caller's own loop: fields in, a step, fields out; a small, flat grid, FS-FD Laplacian
        _case("fs", (256, 64), 3, "f32", 1, lap=2, name="fs2d_256x64_p3_f32_onestep"),
        # a grid of the paper's accuracy table: four order parameters, double precision
        _case("fs", (256, 256), 4, "f64", 40, name="fs2d_256_p4_f64"),
        # the time-to-accuracy workload in double precision
        _case("fs", (1024, 1024), 2, "f64", 8, start="noise", name="fs2d_1024_p2_f64"),
        # the headline workload: a stretch of a long FP32 run
        _case("fs", (1024, 1024), 2, "f32", 100, start="noise", name="fs2d_1024_p2_f32"),
        # the paper's finest 2D grid, four order parameters
        _case("fs", (2048, 2048), 4, "f32", 32, name="fs2d_2048_p4_f32"),
        # a 3D grid of the paper's second table, double precision
        _case("fs", (64, 64, 64), 4, "f64", 16, name="fs3d_64_p4_f64"),
        # the large 3D workload
        _case("fs", (256, 256, 256), 2, "f32", 20, start="noise", name="fs3d_256_p2_f32"),
        # a parameter sweep: many 2D simulations of uneven size in one plan
        _case("ensemble", (0, 0), 2, "f32", 32, members=64, start="noise", name="ensemble_64_p2_f32"),
        # fitting the four parameters to a trajectory: forward, loss, backward
        _case("trajectory", (512, 512), 2, "f32", 20, every=10, name="trajectory_512_p2_f32"),
        # the explicit comparison scheme in 2D, double precision, a flat grid
        _case("fd", (512, 256), 4, "f64", 64, name="fd2d_512x256_p4_f64"),
        # the explicit comparison scheme in 3D, FP32
        _case("fd", (128, 128, 128), 4, "f32", 32, name="fd3d_128_p4_f32"),
    ]


def _case(kind, n, p, precision, steps, lap=0, start="grains", members=1, every=1, name=None):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2] if len(n) > 2 else 1, "p": p, "precision": precision, "lap": lap,
         "steps": steps, "start": start, "members": members, "every": every}
    if name:
        c["name"] = name
    return c


_KINDS = ["fs2", "fs2", "fs2", "fs3", "fs3", "fd2", "fd3", "ensemble", "trajectory", "adjoint2", "adjoint3"]


def draw(rng):
    """One more case of the ranges above.  Axes are powers of two (the library takes no others), drawn each by itself, so most
    grids are not square; p and the step counts take odd values too."""
    kind = rng.choice(_KINDS)
    precision = rng.choice(["f64", "f32"])
    lap = rng.choice([0, 0, 1, 2])
    start = rng.choice(["noise", "grains"])
    p = rng.randint(1, 4)

    def axes(lo, hi, count, most):
        while True:
            n = tuple(1 << rng.randint(lo, hi) for _ in range(count))
            if math.prod(n) <= most:
                return n

    f64 = precision == "f64"
    if kind == "fs2":
        n = axes(6, 11, 2, (1 << 20) if f64 else (1 << 22))
        return _case("fs", n, rng.randint(0, 4), precision, _steps(rng, n, p, f64), lap=lap, start=start)
    if kind == "fs3":
        n = axes(4, 8, 3, (1 << 20) if f64 else (1 << 24))
        return _case("fs", n, p, precision, _steps(rng, n, p, f64), lap=lap, start=start)
    if kind == "fd2":
        n = axes(6, 11, 2, (1 << 21) if f64 else (1 << 22))
        return _case("fd", n, p, precision, _steps(rng, n, p, f64), start=start)
    if kind == "fd3":
        n = axes(4, 8, 3, (1 << 21) if f64 else (1 << 24))
        return _case("fd", n, p, precision, _steps(rng, n, p, f64), start=start)
    if kind == "ensemble":
        return _case("ensemble", (0, 0), p, "f32", rng.randint(1, 48), members=int(round(2 ** rng.uniform(2, 6))), start=start)
    if kind == "trajectory":
        n = axes(6, 9, 2, (1 << 18))
        every = rng.randint(2, 8)
        return _case("trajectory", n, p, precision, every * rng.randint(1, 3), lap=lap, every=every)
    n = axes(6, 10, 2, (1 << 20)) if kind == "adjoint2" else axes(4, 7, 3, (1 << 20))
    return _case("adjoint", n, p, precision, 1, lap=lap)


def _steps(rng, n, p, f64):
    """Steps of a drawn pass: up to 200, fewer where the grid is large (double precision counts twenty-fold)."""
    most = 5e8 / (math.prod(n) * (1 + p) * (20 if f64 else 1))
    return max(1, int(2 ** rng.uniform(0, math.log2(max(1.5, min(200.0, most))))))


def _grid(case):
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _problem(case):
    pr = I.Problem(n=_grid(case), p=case["p"], lap=case["lap"])
    # 5 to 6 times the stable FD step for the noise starts, the step of the accuracy tables for developed fields; half the
    # stable step for the explicit scheme
    dt = I.fd_stable_dt(pr)
    if case["kind"] == "fd":
        dt *= 0.5
    elif case["start"] == "noise":
        dt *= 5.0 if pr.npoints <= 64 * 64 else 6.0
    else:
        dt = 5e-3 if pr.ndim == 2 else min(5e-3, 5.0 * dt)
    return pr.replace(dt=dt)


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _fields(pr, start, gen):
    """Fields of one simulation in double precision.  "noise": uniform noise of +-0.01 about 0.5 in every field, the start of
    a coarsening run.  "grains": developed fields, smooth order parameters between 0 and 1 that share the domain, c about 0.5."""
    shape = (pr.nf,) + pr.shape
    if start == "noise":
        return 0.5 + 0.01 * (2.0 * torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") - 1.0)
    coords = torch.meshgrid(*[torch.arange(m, dtype=torch.float64, device="cuda") * (2.0 * math.pi / m)
                              for m in pr.shape], indexing="ij")
    modes = torch.randint(-3, 4, (pr.nf, 4, len(coords)), generator=gen, device="cuda").cpu().tolist()
    phases = (2.0 * math.pi * torch.rand((pr.nf, 4), generator=gen, dtype=torch.float64, device="cuda")).cpu().tolist()
    waves = []
    for f in range(pr.nf):
        w = torch.zeros(pr.shape, dtype=torch.float64, device="cuda")
        for q in range(4):
            w += torch.cos(sum(k * x for k, x in zip(modes[f][q], coords)) + phases[f][q])
        waves.append(w)
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    out[0] = 0.5 + 0.02 * waves[0]
    if pr.p:
        out[1:] = torch.softmax(torch.stack([torch.zeros_like(waves[0])] + waves[1:]), 0)[1:]
    return out


def _members(case):
    # sizes and parameters of the sweep belong to the case, the fields to the seed
    return I.batch_problems(case["members"], seed=case["members"], p=case["p"])


def _inputs(case, seed):
    """The problems and inputs of a case, rounded to its precision: the same for prepare() and exact()."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * (seed + 1))
    dt = _dtype(case)
    if case["kind"] == "ensemble":
        probs = _members(case)
        return probs, [_fields(pr, case["start"], gen).to(dt) for pr in probs], None
    pr = _problem(case)
    u = _fields(pr, case["start"], gen).to(dt)
    extra = None
    if case["kind"] == "trajectory":
        # the target: other developed fields about the start's, one snapshot for every `every` steps
        count = case["steps"] // case["every"]
        extra = torch.stack([_fields(pr, case["start"], gen).to(dt) for _ in range(count)])
    elif case["kind"] == "adjoint":
        extra = torch.rand(u.shape, generator=gen, dtype=torch.float64, device="cuda").to(dt)
    return pr, u, extra


def prepare(case, seed):
    pr, u, extra = _inputs(case, seed)
    state = {"case": case, "prob": pr, "u": u, "extra": extra}
    if case["kind"] == "trajectory":
        state["theta"] = torch.tensor([pr.M, pr.L, pr.kappa_c, pr.kappa_eta], dtype=_dtype(case))
        return state
    scheme = fs.FS_SCHEME_EXPLICIT_FD if case["kind"] == "fd" else fs.FS_SCHEME_SEMI_IMPLICIT_FS
    state["plan"] = fs.Plan(pr, case["precision"], scheme=scheme)
    if case["kind"] == "ensemble":
        state["out"] = [torch.empty_like(m) for m in u]
        state["plan"].set_fields(u)  # the ensemble's schedule is chosen at its first set_fields
    else:
        state["out"] = torch.empty_like(u)
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "trajectory":
        theta = state["theta"].detach().requires_grad_()
        u0 = state["u"].detach().requires_grad_()
        snaps = adjoint.trajectory(theta, u0, state["prob"], case["precision"], case["steps"], case["every"])
        loss = adjoint.misfit_loss(snaps, state["extra"])
        loss.backward()
        return {"snaps": snaps.detach(), "loss": loss.detach(), "theta": theta.grad, "u0": u0.grad}
    plan = state["plan"]
    if case["kind"] == "adjoint":
        # the sensitivities are sums in the plan's precision, whatever the container
        grad = plan.step_adjoint(state["u"], state["extra"], state["out"])
        return {"lam": state["out"], "grad": torch.tensor(grad, dtype=_dtype(case))}
    plan.set_fields(state["u"])
    plan.step(case["steps"])
    return plan.get_fields(state["out"])


def work(case):
    """A step reads and writes every field once; its operations are the pointwise stage, one inverse and one forward real
    transform for each field (2.5 N log2 N each) and the update of N/2 modes.  An explicit step has the stencils in place of
    the transforms.  A backward pass through the trajectory runs the steps again and one adjoint step for each, which
    transforms five arrays for each field."""
    if case["kind"] == "ensemble":
        probs = _members(case)
        sizes = [pr.npoints for pr in probs]
    else:
        sizes = [case["nx"] * case["ny"] * case["nz"]]
    nf, s = 1 + case["p"], 8 if case["precision"] == "f64" else 4
    total_b = total_f = 0.0
    for n in sizes:
        if case["kind"] == "fd":
            b, f = 2 * nf * s * n, n * (22 * nf + 24 * case["p"] + 6)
        else:
            step_b, step_f = 2 * nf * s * n, n * (5.0 * nf * math.log2(n) + 24 * case["p"] + 4 + 5 * nf)
            adj_b, adj_f = 3 * nf * s * n, n * (12.5 * nf * math.log2(n) + 40 * nf)
            if case["kind"] == "adjoint":
                b, f = adj_b, adj_f
            elif case["kind"] == "trajectory":
                b, f = 2 * step_b + adj_b, 2 * step_f + adj_f
            else:
                b, f = step_b, step_f
        total_b += b * case["steps"]
        total_f += f * case["steps"]
    return {"bytes": total_b, "flops": total_f}


# ---- the same in 64 bits with plain torch --------------------------------------------------------------------------------

def _forces(pr, u):
    c, eta = u[0], u[1:]
    h = (eta ** 3 * (6 * eta ** 2 - 15 * eta + 10)).sum(0)
    s2 = (eta ** 2).sum(0)
    d = pr.c_beta - pr.c_alpha
    fc = 2 * pr.rho2 * (c - pr.c_alpha - d * h)
    q = eta * (1 - eta)
    fe = pr.rho2 * d * (pr.c_beta + pr.c_alpha - 2 * c) * 30 * q ** 2 + \
        pr.w * (2 * q * (1 - 2 * eta) + 4 * pr.alpha * eta * (s2 - eta ** 2))
    return torch.cat([fc[None], fe])


def _k2(pr):
    """|xi|^2 on the bins of rfftn."""
    total = 0.0
    for a, (m, h) in enumerate(zip(pr.shape, tuple(reversed(pr.dx)))):
        freq = torch.fft.rfftfreq if a == pr.ndim - 1 else torch.fft.fftfreq
        xi = 2 * math.pi * freq(m, d=h, dtype=torch.float64, device="cuda")
        if pr.lap == 1:
            k = -2 * (torch.cos(h * xi) - 1) / h ** 2
        elif pr.lap == 2:
            k = -(16 * torch.cos(h * xi) - torch.cos(2 * h * xi) - 15) / (6 * h ** 2)
        else:
            k = xi ** 2
        shape = [1] * pr.ndim
        shape[a] = k.numel()
        total = total + k.reshape(shape)
    return total


def _fs_step(pr, u, k2, theta=None):
    mob, rate, kc, ke = theta if theta is not None else (pr.M, pr.L, pr.kappa_c, pr.kappa_eta)
    dims = tuple(range(-pr.ndim, 0))
    f = _forces(pr, u)
    uh = torch.fft.rfftn(u, dim=dims)
    fh = torch.fft.rfftn(f, dim=dims)
    c = (uh[:1] - mob * pr.dt * k2 * fh[:1]) / (1 + mob * pr.dt * kc * k2 ** 2)
    e = (uh[1:] - rate * pr.dt * fh[1:]) / (1 + rate * pr.dt * ke * k2)
    return torch.fft.irfftn(torch.cat([c, e]), s=pr.shape, dim=dims)


def _laplacian(pr, x):
    out = torch.zeros_like(x)
    for a, h in zip(range(-pr.ndim, 0), tuple(reversed(pr.dx))):
        out += (x.roll(1, a) + x.roll(-1, a) - 2 * x) / h ** 2
    return out


def _fd_step(pr, u):
    f = _forces(pr, u)
    mu = f[0] - pr.kappa_c * _laplacian(pr, u[0])
    out = torch.empty_like(u)
    out[0] = u[0] + pr.dt * pr.M * _laplacian(pr, mu)
    out[1:] = u[1:] - pr.dt * pr.L * (f[1:] - pr.kappa_eta * _laplacian(pr, u[1:]))
    return out


def exact(case, seed):
    pr, u, extra = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ensemble":
        return [_advance(q, v.double(), case["steps"]) for q, v in zip(pr, u)]
    u = u.double()
    if kind == "fs":
        return _advance(pr, u, case["steps"])
    if kind == "fd":
        for _ in range(case["steps"]):
            u = _fd_step(pr, u)
        return u
    k2 = _k2(pr)
    theta = torch.tensor([pr.M, pr.L, pr.kappa_c, pr.kappa_eta], dtype=torch.float64, device="cuda").requires_grad_()
    u.requires_grad_()
    if kind == "adjoint":
        (_fs_step(pr, u, k2, theta) * extra.double()).sum().backward()
        return {"lam": u.grad, "grad": theta.grad}
    v, snaps = u, []
    for i in range(case["steps"]):
        v = _fs_step(pr, v, k2, theta)
        if (i + 1) % case["every"] == 0:
            snaps.append(v)
    snaps = torch.stack(snaps)
    loss = ((snaps - extra.double()) ** 2).sum() / math.prod(pr.shape)
    loss.backward()
    return {"snaps": snaps.detach(), "loss": loss.detach(), "theta": theta.grad, "u0": u.grad}


def _advance(pr, u, steps):
    k2 = _k2(pr)
    for _ in range(steps):
        u = _fs_step(pr, u, k2)
    return u
