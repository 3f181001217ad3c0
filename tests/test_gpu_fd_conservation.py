"""The Laplacians of the explicit scheme are nothing on a uniform field: a
uniform state keeps its c bit for bit, however small c is against mu (a residue r
of the stencil weights' sum would move it by r mu in every step: 1e-9 in FP32
against the 6e-11 of a last place of c = 1e-3), and its eta where f_chem is 0."""
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


@pytest.mark.parametrize("precision,c0", [("f32", 1e-3), ("f64", 1e-9)])
@pytest.mark.parametrize("p", [0, 2])
@pytest.mark.parametrize("n,dx", [((64, 16), (1.0, 0.8)), ((32, 32), (0.7, 0.7)), ((8, 16, 8), (1.0, 1.0, 1.0)),
                                  ((16, 8, 8), (1.0, 0.8, 0.9))])
def test_uniform_state_keeps_c(F, n, dx, p, precision, c0):
    import torch
    pr = I.Problem(n=n, dx=dx, p=p)
    pr.dt = 0.9 * I.fd_stable_dt(pr)
    f0 = np.full((1 + p,) + pr.shape, 0.25)
    f0[0] = c0
    t = torch.tensor(f0, dtype=torch.float32 if precision == "f32" else torch.float64, device="cuda")
    plan = F.Plan(pr, precision, scheme=F.FS_SCHEME_EXPLICIT_FD)
    plan.set_fields(t)
    plan.step(50)
    got = plan.get_fields()
    plan.close()
    assert torch.equal(got[0], t[0]), float((got[0].double() - t[0].double()).abs().max())


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n,dx", [((64, 16), (1.0, 0.8)), ((16, 8, 8), (1.0, 0.8, 0.9)), ((8, 16, 8), (1.0, 1.0, 1.0))])
def test_uniform_state_without_reaction_stays(F, n, dx, precision):
    """f_chem = 0: only the Laplacians are left, nothing on a uniform state at
    any dt (a stencil that rounds its centre apart moves it at a large one)."""
    import torch
    pr = I.Problem(n=n, dx=dx, p=3, rho2=0.0, w=0.0)
    pr.dt = 1000.0
    t = torch.full((4,) + pr.shape, 0.3, dtype=torch.float32 if precision == "f32" else torch.float64, device="cuda")
    plan = F.Plan(pr, precision, scheme=F.FS_SCHEME_EXPLICIT_FD)
    plan.set_fields(t)
    plan.step(3)
    got = plan.get_fields()
    plan.close()
    assert torch.equal(got, t), float((got.double() - t.double()).abs().max())


@pytest.mark.parametrize("n,dx", [((64, 64), (1.0, 0.8)), ((32, 32, 32), (1.0, 0.8, 0.9))])
def test_mean_of_c_over_many_steps_fp32(F, n, dx):
    """p = 0, noise, to rest: every step rounds c once (at most 2^-25 at c in
    [1/4, 1/2)), and the mean of N such errors, taken as independent while the
    field still moves and absent once it rests, is of order 2^-25 sqrt(steps / N);
    2e-7 allows four times the worst of both grids' 2^-25 sqrt(2000 / 4096) and a
    last place of the mean.  Weights that sum to 1e-9 lose 1e-9 |mu| 2000 = 1e-6."""
    import torch
    pr = I.Problem(n=n, dx=dx, p=0)
    pr.dt = 0.9 * I.fd_stable_dt(pr)
    f0 = I.noise_fields(pr, seed=5, c0=0.4, amp=0.05)
    t = torch.tensor(f0, dtype=torch.float32, device="cuda")
    plan = F.Plan(pr, "f32", scheme=F.FS_SCHEME_EXPLICIT_FD)
    plan.set_fields(t)
    plan.step(2000)
    got = plan.get_fields()
    plan.close()
    assert abs(float(got[0].double().mean() - t[0].double().mean())) <= 2e-7
