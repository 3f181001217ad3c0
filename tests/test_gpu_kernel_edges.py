"""The kernels at the sizes where they can go wrong: shortest and longest
lines, single tiles, odd numbers of order parameters, remainders of tiles,
denominators beyond the reciprocal's range -- against the FP64 oracle.

Tolerances (relative L-inf per field), as in the other parity tests: FP64
transforms and updates of O(1) data, 1e-12 per step; FP32 2e-6 per step and a
factor 2 over several steps; adjoint 1e-11 (FP64) and 2e-5 (FP32) for the
field, ten times that of the largest for the four sums."""
import numpy as np
import pytest

from paper_2306_04322_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_04322_gb300 import build as B
    from paper_2306_04322_gb300 import fs
    B.build()
    fs.lib()
    return fs


def rel_linf(a, b):
    return max(np.max(np.abs(a[f] - b[f])) / max(np.max(np.abs(b[f])), 1e-300) for f in range(b.shape[0]))


def dtype(precision):
    import torch
    return torch.float64 if precision == "f64" else torch.float32


def tol(precision, k):
    return 1e-12 * k if precision == "f64" else 2e-6 * k * (2.0 if k > 1 else 1.0)


def problem(n, p, **kw):
    pr = I.Problem(n=n, p=p, **kw)
    pr.dt = 5.0 * I.fd_stable_dt(pr)
    return pr


def check_steps(F, O, pr, precision, forms=(0, 0), scheme=None):
    """One step (from the real fields), then four more, each read back."""
    import torch
    f0 = I.noise_fields(pr, seed=31)
    kw = {} if scheme is None else {"scheme": scheme}
    plan = F.Plan(pr, precision, **kw)
    if forms != (0, 0):
        F.fs_set_pass_forms(plan.h, *forms)
    t0 = torch.tensor(f0, dtype=dtype(precision), device="cuda")
    plan.set_fields(t0)
    ref = t0.double().cpu().numpy()
    out = []
    for k, n in ((1, 1), (5, 4)):
        plan.step(n)
        got = plan.get_fields().double().cpu().numpy()
        ref = O.fd_step(pr, ref, n) if scheme is not None else O.step(pr, ref, n)[0]
        assert rel_linf(got, ref) <= tol(precision, k), (k, rel_linf(got, ref))
        out.append(got)
    plan.close()
    return out


@pytest.mark.parametrize("n,p", [
    ((64, 64), 0), ((64, 64), 4), ((128, 64), 3), ((64, 128), 1), ((256, 128), 2), ((128, 256), 4), ((512, 64), 0),
    ((64, 512), 3), ((256, 512), 2), ((1024, 64), 4), ((64, 1024), 1), ((2048, 64), 2), ((64, 2048), 3),
    ((32, 2048), 0), ((2048, 8), 4), ((8, 64), 2), ((16, 1024), 1), ((512, 8, 8), 1), ((64, 8, 16), 4),
    ((8, 64, 64), 2), ((128, 16, 8), 0), ((1024, 8, 8), 3)])
def test_fp64_pair_rows_and_columns(F, O, n, p):
    """Pair-form rows, single-column units, their mix with the other forms on
    axes that have only one of them, and both against form 1."""
    pr = problem(n, p)
    a = check_steps(F, O, pr, "f64")
    b = check_steps(F, O, pr, "f64", forms=(1, 1))
    for x, y in zip(a, b):
        assert rel_linf(x, y) <= 1e-11


@pytest.mark.parametrize("kappa", [1e305, 1e308])
@pytest.mark.parametrize("n", [(64, 64), (16, 16), (16, 16, 16)])
def test_fp64_update_with_denominators_out_of_the_reciprocals_range(F, O, n, kappa):
    """1 + M dt kappa k^4 from 1 (k = 0) to beyond 2^1009 and to infinity:
    the modes go to zero as the division's do."""
    pr = I.Problem(n=n, p=2, kappa_c=kappa, kappa_eta=kappa)
    pr.dt = 1e-2
    check_steps(F, O, pr, "f64")


@pytest.mark.parametrize("n,p", [
    # four-column tiles: one, two and many blocks, with and without eta, odd p; pairs below 16 rows' points
    ((8, 64), 2), ((16, 64), 1), ((16, 128), 4), ((32, 256), 3), ((16, 512), 2), ((8, 1024), 1), ((16, 1024), 3),
    ((512, 1024), 1), ((1024, 1024), 0), ((1024, 1024), 1), ((1024, 1024), 3), ((2048, 1024), 4), ((16, 2048), 2),
    ((8, 2048), 1), ((2048, 128), 1), ((2048, 64), 1),
    # several row pairs per CTA of an x pass, 2D and 3D
    ((64, 2048), 2), ((128, 2048), 0), ((256, 1024), 3), ((256, 1024), 4),
    ((64, 8, 8), 0), ((64, 16, 16), 3), ((64, 128, 128), 2), ((128, 8, 8), 4), ((128, 64, 64), 1), ((256, 8, 8), 2),
    ((256, 32, 64), 3), ((512, 8, 8), 1), ((512, 16, 64), 4),
    # y / z lines on fewer columns than a tile has
    ((8, 64, 32), 1), ((16, 256, 8), 2), ((8, 8, 256), 0)])
def test_fp32_column_tiles_and_row_groups(F, O, n, p):
    check_steps(F, O, problem(n, p), "f32")


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n,p", [
    ((8, 8), 4), ((8, 64), 1), ((64, 8), 2), ((2048, 8), 0), ((8, 2048), 3), ((512, 32), 4), ((8, 8, 8), 2),
    ((8, 64, 8), 4), ((64, 8, 16), 0), ((16, 8, 128), 3), ((256, 16, 8), 1)])
def test_fd_tiles_and_their_remainders(F, O, n, p, precision):
    pr = I.Problem(n=n, p=p, dx=(1.0, 0.5, 2.0)[:len(n)])
    pr.dt = 0.9 * I.fd_stable_dt(pr)
    check_steps(F, O, pr, precision, scheme=F.FS_SCHEME_EXPLICIT_FD)


@pytest.mark.parametrize("n", [(64, 16), (16, 8, 16)])
@pytest.mark.parametrize("field,value", [(0, np.nan), (1, np.inf), (2, -np.inf)])
def test_fd_reports_a_nonfinite_point(F, n, field, value):
    import torch
    pr = I.Problem(n=n, p=2)
    pr.dt = 0.5 * I.fd_stable_dt(pr)
    f0 = I.noise_fields(pr, seed=3)
    f0.reshape(3, -1)[field, -1] = value
    plan = F.Plan(pr, "f32", scheme=F.FS_SCHEME_EXPLICIT_FD)
    plan.set_fields(torch.tensor(f0, dtype=torch.float32, device="cuda"))
    with pytest.raises(F.FSError) as ei:
        plan.step(1)
    assert ei.value.status == F.FS_ERR_NONFINITE
    plan.close()


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n,p", [((8, 8), 1), ((8, 64), 4), ((64, 8), 3), ((1024, 8), 2), ((16, 1024), 0),
                                 ((256, 512), 4), ((8, 8, 8), 4), ((128, 8, 8), 1), ((8, 16, 64), 3)])
def test_adjoint_tiles(F, O, n, p, precision):
    import torch
    pr = problem(n, p)
    rng = np.random.default_rng(12)
    u = torch.tensor(I.noise_fields(pr, seed=61, amp=0.3), dtype=dtype(precision), device="cuda")
    lam = torch.tensor(rng.standard_normal(tuple(u.shape)), dtype=dtype(precision), device="cuda")
    out = torch.empty_like(lam)
    plan = F.Plan(pr, precision)
    grad = np.array(plan.step_adjoint(u, lam, out))
    plan.close()
    ref, gref = O.adjoint_step(pr, u.double().cpu().numpy(), lam.double().cpu().numpy())
    t = 1e-11 if precision == "f64" else 2e-5
    assert rel_linf(out.double().cpu().numpy(), ref) <= t
    assert np.max(np.abs(grad - gref)) <= 10 * t * np.max(np.abs(gref))


@pytest.mark.parametrize("precision,p,sizes", [
    ("f32", 0, [(64, 128), (1024, 128), (64, 512)]),
    ("f32", 3, [(64, 1024), (128, 128), (512, 256), (64, 128)]),
    ("f32", 4, [(16, 512), (32, 512), (128, 128)]),     # members that only form 1 covers
    ("f64", 1, [(64, 64), (16, 1024), (256, 64)])])
def test_ensemble_items(F, O, precision, p, sizes):
    import torch
    probs = [problem(n, p) for n in sizes]
    fields = [torch.tensor(I.noise_fields(pr, seed=70 + i), dtype=dtype(precision), device="cuda")
              for i, pr in enumerate(probs)]
    plan = F.Plan(probs, precision)
    plan.set_fields(fields)
    plan.step(3)
    got = [o.double().cpu().numpy() for o in plan.get_fields()]
    plan.close()
    for pr, f, g in zip(probs, fields, got):
        ref, _ = O.step(pr, f.double().cpu().numpy(), 3)
        assert rel_linf(g, ref) <= tol(precision, 3)
