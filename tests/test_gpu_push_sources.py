"""Pushes of memory that a kernel of the plan's device must not read with its
own loads (odd addresses; host memory that the caller names device memory) hold
the pixels that were pushed: the runtime copies them."""
import ctypes

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


@pytest.mark.parametrize("source", ["odd", "even", "pinned"])
@pytest.mark.parametrize("nx,extra", [(333, 0), (333, 5), (384, 0)])   # (384: rows fill the pitch)
@pytest.mark.parametrize("block", [False, True])
def test_pushed_pixels(source, nx, extra, block):
    L, ny, rp = 4, 77, nx + extra
    size = L * ny * rp * 2
    g = torch.Generator().manual_seed(nx + extra)
    raw = torch.randint(0, 100, (size + 2,), generator=g, dtype=torch.uint8)
    raw = raw.pin_memory() if source == "pinned" else raw.cuda()
    at = 1 if source == "odd" else 2
    want = raw[at:at + size].cpu().numpy().view("<i2").reshape(L, ny, rp)[:, :, :nx]
    lib = F.load()
    with F.Plan(nx, ny, L, 5, 6.0, F.BRANCH_IMAGE, F.F16) as p:
        torch.cuda.synchronize()
        if block:
            assert lib.fitrig_push_snapshots(p.h, ctypes.c_void_p(raw.data_ptr() + at), L, F.F16, 1,
                                             rp, 0) == F.OK
        else:
            for s in range(L):
                ptr = ctypes.c_void_p(raw.data_ptr() + at + s * ny * rp * 2)
                assert lib.fitrig_push_snapshot(p.h, ptr, F.F16, 1, rp) == F.OK
        torch.cuda.synchronize()
        for s in range(L):
            ptr, pitch = F.fitrig_stack_device_ptr(p.h, s)
            got = torch.as_tensor(_Dev(ptr, (ny, pitch), "<i2"), device="cuda")[:, :nx]
            assert (got.cpu().numpy() == want[s]).all()
