"""Pushes of snapshots whose rows do not fill the device pitch: the staged
host copies and the one-copy blocks hold the pixels that were pushed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402


class _Dev:
    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr,
                                         "version": 2, "strides": None}


# row bytes divisible by 16, 8, 4 and 2 only, by 128 (no staging), snapshots on
# both sides of the staging's least size and of a slot's rows
@pytest.mark.parametrize("dtype,nx,ny", [(torch.float32, 1004, 1100), (torch.float32, 1002, 1100),
                                         (torch.float32, 1001, 1100), (torch.bfloat16, 2001, 1100),
                                         (torch.float32, 1024, 1100), (torch.float32, 1001, 400),
                                         (torch.float16, 3001, 1500)])
@pytest.mark.parametrize("source", ["pinned", "pageable", "device"])
@pytest.mark.parametrize("block", [False, True])
def test_pushed_pixels(dtype, nx, ny, source, block):
    L = 5
    storage = {torch.float32: F.F32, torch.bfloat16: F.BF16, torch.float16: F.F16}[dtype]
    g = torch.Generator(device="cuda").manual_seed(nx)
    x = torch.randn(L, ny, nx, device="cuda", generator=g).to(dtype)
    src = x if source == "device" else x.cpu().pin_memory() if source == "pinned" else x.cpu()
    with F.Plan(nx, ny, L, 5, 6.0, F.BRANCH_IMAGE, storage) as p:
        for _ in range(2):                # a plan is filled again after a reset
            F.fitrig_plan_reset(p.h)
            if block:
                F.fitrig_push_snapshots(p.h, src[:2])
                F.fitrig_push_snapshots(p.h, src[2:])
            else:
                p.push_stack(src)
            torch.cuda.synchronize()
            for s in range(L):
                ptr, pitch = F.fitrig_stack_device_ptr(p.h, s)
                kind = "<f4" if dtype == torch.float32 else "<i2"
                got = torch.as_tensor(_Dev(ptr, (ny, pitch), kind), device="cuda")[:, :nx]
                want = x[s] if dtype == torch.float32 else x[s].view(torch.int16)
                assert torch.equal(got, want)
