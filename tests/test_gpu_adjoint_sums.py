"""The four sensitivities of an adjoint step.

FP32: their rounding is pinned.  The sums can cancel to a hundredth of their
terms, so their last digits are those of the transforms and of f(u); a caller
who fits parameters gets the same digits from build to build
(tests/golden/adjoint_fp32_sensitivities.txt).  What may differ is the order of
the FP64 sums: at most 2^17 terms of a few times the result each,
2^17 2^-53 10 = 1.5e-10 of the largest entry.  One FP32 rounding more or less in a
transform moves an entry by 1e-8 or more."""
import os

import numpy as np
import pytest

from paper_2306_04322_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "adjoint_fp32_sensitivities.txt")


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


def golden_rows():
    rows = []
    with open(GOLDEN) as f:
        for line in f:
            if line.strip() and not line.startswith("#"):
                w = line.split()
                rows.append((tuple(int(v) for v in w[0].split("x")), int(w[1]), int(w[2]), [float(v) for v in w[3:7]]))
    return rows


def problem(n, p, lap=0):
    pr = I.Problem(n=n, p=p, lap=lap)
    pr.dt = 5.0 * I.fd_stable_dt(pr)
    return pr


def state(pr):
    """u about 0.5 +- 0.3, lam' uniform in (0, 1): as the misfit of two states, with a mean."""
    return I.noise_fields(pr, seed=81, amp=0.3), I.noise_fields(pr, seed=82, amp=0.5)


def sums(F, pr, u, lam, precision):
    import torch
    dt = torch.float64 if precision == "f64" else torch.float32
    plan = F.Plan(pr, precision)
    ut, lt = (torch.tensor(v, dtype=dt, device="cuda") for v in (u, lam))
    out = torch.empty_like(lt)
    g = np.array(plan.step_adjoint(ut, lt, out))
    plan.close()
    return g, ut.double().cpu().numpy(), lt.double().cpu().numpy()


@pytest.mark.parametrize("n,p,lap,want", golden_rows())
def test_fp32_sums_keep_their_digits(F, n, p, lap, want):
    pr = problem(n, p, lap)
    got, _, _ = sums(F, pr, *state(pr), "f32")
    assert np.max(np.abs(got - want)) <= 1.5e-10 * np.max(np.abs(want)), (got, want)


@pytest.mark.parametrize("n", [(32, 64), (16, 8, 32)])
@pytest.mark.parametrize("exponent", [-100, 110])
def test_fp32_sums_scale_with_the_cotangent(F, n, exponent):
    """A power of two on lam' is one on the sums, over the FP32 range of lam'
    and its transform (lam'^ up to 2^122, products beyond FP32)."""
    pr = problem(n, 2)
    u, lam = state(pr)
    lam = lam.astype(np.float32)
    base, _, _ = sums(F, pr, u, lam, "f32")
    got, _, _ = sums(F, pr, u, lam * np.float32(2.0 ** exponent), "f32")
    # 1e-9: lam'^ below 2^-126 + 24 keeps fewer bits
    assert np.all(np.abs(got * 2.0 ** -exponent - base) <= 1e-9 * np.max(np.abs(base))), (got * 2.0 ** -exponent, base)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n,p", [((64, 64), 1), ((1024, 8), 2), ((256, 512), 4), ((16, 1024), 3), ((8, 16, 64), 3),
                                 ((128, 8, 8), 1)])
def test_each_sum_to_its_own_scale(F, O, n, p, precision):
    """g_q = (1/N) sum_k conj(lam'^) (dD1_q u^ + dD2_q f^): with transforms of
    relative error e in the 2-norm (2e-6 FP32, the bound of a step; 1e-12 FP64)
    the error of g_q is at most e (|dD1 lam'^| |u^| + |dD2 lam'^| |f^| +
    |lam'^| (|dD1 u^| + |dD2 f^|)) / N, summed over the fields q acts on."""
    pr = problem(n, p)
    got, u, lam = sums(F, pr, *state(pr), precision)
    _, ref = O.adjoint_step(pr, u, lam)
    axes = tuple(range(1, u.ndim))
    uh, lh, fh = (np.fft.fftn(v, axes=axes) for v in (u, lam, O.derivatives(pr, u)))
    k2, e, N = O.k2(pr), 2e-6 if precision == "f32" else 1e-12, pr.npoints
    norm = lambda v: float(np.sqrt(np.sum(np.abs(v) ** 2)))
    for q, (rate, kap, fields) in enumerate(((pr.M, pr.kappa_c, [0]), (pr.L, pr.kappa_eta, range(1, p + 1)),
                                             (pr.M, pr.kappa_c, [0]), (pr.L, pr.kappa_eta, range(1, p + 1)))):
        m, kk = (k2, k2 * k2) if fields == [0] else (np.ones_like(k2), k2)
        i2 = 1.0 / (1.0 + rate * pr.dt * kap * kk) ** 2
        d1, d2 = (-pr.dt * kap * kk * i2, -pr.dt * m * i2) if q < 2 else \
            (-rate * pr.dt * kk * i2, (rate * pr.dt) ** 2 * kk * m * i2)
        value = sum(np.sum(lh[f].conj() * (d1 * uh[f] + d2 * fh[f])).real for f in fields) / N
        assert abs(value - ref[q]) <= 1e-9 * np.max(np.abs(ref))  # the same formula as the oracle's
        bound = e / N * sum(norm(d1 * lh[f]) * norm(uh[f]) + norm(d2 * lh[f]) * norm(fh[f]) +
                            norm(lh[f]) * (norm(d1 * uh[f]) + norm(d2 * fh[f])) for f in fields)
        assert abs(got[q] - ref[q]) <= bound, (q, got[q], ref[q], bound)
