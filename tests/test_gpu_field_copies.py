"""The caller's field pointers: fields of one allocation in order, out of order
or with gaps, fields in allocations that happen to be neighbours in the address
space, and host arrays.  Every value comes back, bit for bit, and an adjoint step
does not depend on where its fields lie."""
import ctypes

import numpy as np
import pytest

from paper_2306_04322_gb300 import inputs as I

pytestmark = pytest.mark.gpu
N, NF = (1024, 512), 3          # 2 MiB a field in FP32: a whole page of the device's allocator
BYTES = 4 * N[0] * N[1]


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


class DeviceBlocks:
    """Separate device allocations of one field each, in address order."""

    def __init__(self, count):
        import torch
        torch.zeros(1, device="cuda")  # the primary context
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.cu.cuMemAlloc_v2.argtypes = [ctypes.POINTER(ctypes.c_uint64), ctypes.c_size_t]
        self.cu.cuMemFree_v2.argtypes = [ctypes.c_uint64]
        self.ptrs = []
        for _ in range(count):
            p = ctypes.c_uint64()
            assert self.cu.cuMemAlloc_v2(ctypes.byref(p), BYTES) == 0
            self.ptrs.append(p.value)
        self.ptrs.sort()

    def neighbours(self, count):
        for i in range(len(self.ptrs) - count + 1):
            if all(self.ptrs[i + k] == self.ptrs[i] + k * BYTES for k in range(count)):
                return self.ptrs[i:i + count]
        return None

    def free(self):
        import torch
        torch.cuda.synchronize()
        for p in self.ptrs:
            self.cu.cuMemFree_v2(p)


def problem():
    pr = I.Problem(n=N, p=NF - 1)
    pr.dt = 5.0 * I.fd_stable_dt(pr)
    return pr


def layouts(kind):
    """nf pointers and what keeps their memory."""
    import torch
    if kind == "in order":
        t = torch.empty((NF,) + N[::-1], device="cuda")
        return [t[f] for f in range(NF)], t
    if kind == "reversed":
        t = torch.empty((NF,) + N[::-1], device="cuda")
        return [t[NF - 1 - f] for f in range(NF)], t
    if kind == "gaps":
        t = torch.empty((2 * NF,) + N[::-1], device="cuda")
        return [t[0], t[1], t[4]], t
    if kind == "host":
        a = np.empty((NF,) + N[::-1], dtype=np.float32)
        return [a[f] for f in range(NF)], a
    if kind == "pinned":
        t = torch.empty((NF,) + N[::-1]).pin_memory()
        return [t[f] for f in range(NF)], t
    b = DeviceBlocks(24)
    ptrs = b.neighbours(NF)
    if ptrs is None:
        b.free()
        pytest.skip("no neighbouring allocations on this device")
    return ptrs, b


@pytest.mark.parametrize("kind", ["in order", "reversed", "gaps", "host", "pinned", "neighbours"])
def test_fields_in_and_out(F, kind):
    import torch
    pr = problem()
    f0 = I.noise_fields(pr, seed=3).astype(np.float32)
    src = torch.tensor(f0, device="cuda")
    plan = F.Plan(pr, "f32")
    dst, keep = layouts(kind)
    plan.set_fields(src)
    F.fs_get_fields(plan.h, dst)      # out to the layout
    plan.set_fields(torch.zeros_like(src))
    F.fs_set_fields(plan.h, dst)      # in from it
    back = plan.get_fields()
    plan.close()
    if isinstance(keep, DeviceBlocks):
        keep.free()
    assert torch.equal(back.cpu(), torch.tensor(f0))


@pytest.mark.parametrize("kind", ["reversed", "gaps", "host", "neighbours"])
def test_adjoint_step_from_any_layout(F, kind):
    import torch
    pr = problem()
    u = torch.tensor(I.noise_fields(pr, seed=4, amp=0.3), dtype=torch.float32, device="cuda")
    lam = torch.tensor(I.noise_fields(pr, seed=5, amp=0.5), dtype=torch.float32, device="cuda")
    out = torch.empty_like(lam)
    plan = F.Plan(pr, "f32")
    want = plan.step_adjoint(u, lam, out)
    dst, keep = layouts(kind)
    plan.set_fields(lam)
    F.fs_get_fields(plan.h, dst)      # lam' in the layout, lambda over it
    got = F.fs_step_adjoint(plan.h, [u[f] for f in range(NF)], dst, dst)
    torch.cuda.synchronize()
    F.fs_set_fields(plan.h, dst)
    back = plan.get_fields()
    plan.close()
    if isinstance(keep, DeviceBlocks):
        keep.free()
    assert torch.equal(back, out)
    # FP64 sums in another order
    assert np.max(np.abs(np.array(got) - np.array(want))) <= 1e-12 * np.max(np.abs(want))
