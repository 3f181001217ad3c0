"""Sums over CTAs of 4 to 16 threads (short axes): the free energy and the four
sensitivities of an adjoint step, against the FP64 oracle.  Which lanes a CTA
has: min(nx / 2, tile) columns x (line / values per thread).  Tolerances: a sum of
at most 4096 FP64 terms, each of FP64 transforms (1e-12) or FP32 ones (2e-6 of
the sum of its parts, all positive, for the energy; the bound of
test_gpu_adjoint_sums for the sensitivities)."""
import numpy as np
import pytest

from paper_2306_04322_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GRIDS = [(8, 8), (8, 16), (16, 8), (8, 8, 8), (16, 8, 8), (8, 16, 8), (8, 8, 16), (8, 8, 32), (16, 16, 16), (32, 8, 8)]


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


@pytest.mark.parametrize("precision,tol", [("f64", 1e-12), ("f32", 4e-6)])
@pytest.mark.parametrize("n", GRIDS)
def test_free_energy_of_small_grids(F, O, n, precision, tol):
    import torch
    pr = I.Problem(n=n, p=2)
    pr.dt = 5.0 * I.fd_stable_dt(pr)
    f0 = torch.tensor(I.noise_fields(pr, seed=17, amp=0.3), device="cuda",
                      dtype=torch.float64 if precision == "f64" else torch.float32)
    plan = F.Plan(pr, precision)
    plan.set_fields(f0)
    got, parts = plan.free_energy()
    plan.close()
    want, ref = O.free_energy(pr, f0.double().cpu().numpy(), parts=True)
    assert abs(got - want) <= tol * abs(want)
    assert np.max(np.abs(np.array(parts)[:len(ref)] - np.array(ref))) <= tol * abs(want)


@pytest.mark.parametrize("precision,tol", [("f64", 1e-11), ("f32", 2e-5)])
@pytest.mark.parametrize("n", GRIDS)
def test_adjoint_sums_of_small_grids(F, O, n, precision, tol):
    import torch
    pr = I.Problem(n=n, p=2)
    pr.dt = 5.0 * I.fd_stable_dt(pr)
    dt = torch.float64 if precision == "f64" else torch.float32
    u = torch.tensor(I.noise_fields(pr, seed=18, amp=0.3), dtype=dt, device="cuda")
    lam = torch.tensor(I.noise_fields(pr, seed=19, amp=0.5), dtype=dt, device="cuda")
    out = torch.empty_like(lam)
    plan = F.Plan(pr, precision)
    g = np.array(plan.step_adjoint(u, lam, out))
    plan.close()
    ref, gref = O.adjoint_step(pr, u.double().cpu().numpy(), lam.double().cpu().numpy())
    # M and kappa_c, L and kappa_eta: each pair to the larger of its own
    for pair in ([0, 2], [1, 3]):
        assert np.max(np.abs(g - gref)[pair]) <= tol * np.max(np.abs(gref[pair])) * (1 if precision == "f64" else 10)
    assert np.max(np.abs(out.double().cpu().numpy() - ref)) <= tol * np.max(np.abs(ref))
