"""Rounding of the steps' transforms and of the FP64 quotient.

Transforms: with M = L = 0 a step is the transform forward and back and a
division by N.  Rounding model: in each of the S = 2 log2(N) radix-2 stages every
value is rounded once as a sum, and half of the values once more as a product (a
whole one is allowed for), each rounding a relative error of 0.425 units (units
of 2^-53, FP32 2^-24: uniform in a last place, logarithmic mantissas): 0.425
sqrt(2 S).  A butterfly that rounds twice at the size of its sum, or the product
in two steps, takes 0.425 sqrt(2.5 S) and more.  4096 values or more per grid
make the measured rms good to 2 %.

Quotient: the reciprocal of KUpdate::quot is rounded to 0.5 + 2^-7 of a last
place (e^3 = 2^-60), so it differs from the rounded quotient only next to ties,
in at most 2 2^-7 of all cases, and never by more than a last place."""
import ctypes
import os
import subprocess

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


@pytest.mark.parametrize("forms", [(0, 0), (1, 1)])
@pytest.mark.parametrize("precision,n", [
    ("f64", (64, 64)), ("f64", (128, 128)), ("f64", (256, 256)), ("f64", (512, 64)), ("f64", (64, 1024)), ("f64", (128, 32, 64)),
    ("f32", (64, 64)), ("f32", (256, 256)), ("f32", (1024, 128)), ("f32", (128, 2048)), ("f32", (64, 64, 64)),
    ("f32", (256, 16, 128))])
def test_transform_forward_and_back(F, precision, n, forms):
    import torch
    pr = I.Problem(n=n, p=1, M=0.0, L=0.0)
    pr.dt = 1e-2
    f = 2.0 * (I.noise_fields(pr, seed=9, amp=1.0) - 0.5)
    f -= f.mean()
    t = torch.tensor(f, dtype=torch.float64 if precision == "f64" else torch.float32, device="cuda")
    plan = F.Plan(pr, precision)
    if forms != (0, 0):
        F.fs_set_pass_forms(plan.h, *forms)
    plan.set_fields(t)
    plan.step(1)
    e = plan.get_fields().double() - t.double()
    plan.close()
    unit = 2.0 ** -53 if precision == "f64" else 2.0 ** -24
    rms = float(e.norm() / t.double().norm()) / unit
    bound = 0.425 * np.sqrt(2 * 2 * np.log2(pr.npoints))
    assert rms <= bound, (rms, bound)


def test_fp64_quotient(F, tmp_path):
    from paper_2306_04322_gb300 import build as B
    src = tmp_path / "quot.cu"
    src.write_text("""#include "fs_kernels.cuh"
__global__ void q(double x, const double* y, double* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = fs::KUpdate<double>::quot(x, y[i]);
}
extern "C" __attribute__((visibility("default"))) int quot(double x, const double* y, double* r, int n) {
  q<<<(n + 255) / 256, 256>>>(x, y, r, n);
  return (int)cudaDeviceSynchronize();
}
""")
    lib = tmp_path / "quot.so"
    subprocess.run([B.nvcc()] + B.ARCH + B.FLAGS + ["-shared", str(src), "-o", str(lib)], check=True,
                   stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    import torch
    call = ctypes.CDLL(os.fspath(lib)).quot
    call.argtypes = [ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    rng = np.random.default_rng(4)
    y = np.concatenate([[1.0, 2.0, 2.0 ** 1008, np.nextafter(1.0, 2.0), 1e305, 1.7e308, np.inf],
                        np.exp(rng.uniform(0.0, 20.0, 1 << 18)), np.exp(rng.uniform(0.0, 690.0, 1 << 18))])
    yt = torch.tensor(y, device="cuda")
    for x in (2.0 ** -21, 1.0):
        r = torch.empty_like(yt)
        torch.cuda.synchronize()
        assert call(x, yt.data_ptr(), r.data_ptr(), len(y)) == 0
        got, want = r.cpu().numpy(), x / y
        off = np.abs(got - want)
        assert np.all(off <= np.spacing(want))
        assert np.mean(off > 0) <= 2.0 ** -6
