"""Host pushes whose rows do not fill the device pitch are staged in memory that
the plan has anyway, or, where its candidate buffers are small, in no more than
the push: the device memory that plans hold, and the pixels."""
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


# candidate buffers of 5.6 MB a unit (the push fits), 35 KB and 32 KB (it does not)
@pytest.mark.parametrize("ny,nx,w,cap,held", [(1100, 1001, 2, 0, 0), (1100, 1001, 32, 0, 1),
                                              (1100, 1001, 5, 1000, 1)])
@pytest.mark.parametrize("block", [False, True])
def test_memory_of_plans_and_pixels(ny, nx, w, cap, held, block):
    L, plans = 4, 6
    x = torch.randn(L, ny, nx, generator=torch.Generator().manual_seed(w)).pin_memory()
    dev = x.cuda()
    ps = []
    try:
        for _ in range(plans):
            p = F.Plan(nx, ny, L, w, 6.0, F.BRANCH_IMAGE, max_selected=cap)
            ps.append(p)
            p.push_stack(dev)   # the plan's memory is there
            F.fitrig_plan_reset(p.h)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for p in ps:
            if block:
                F.fitrig_push_snapshots(p.h, x)
            else:
                p.push_stack(x)
        push = x.numel() * 4 if block else x[0].numel() * 4
        # (2 MB: what an allocation is rounded to; 16 MB: streams and events)
        assert free - torch.cuda.mem_get_info()[0] <= plans * held * (push + (2 << 20)) + (16 << 20)
        for p in ps:
            for s in range(L):
                ptr, pitch = F.fitrig_stack_device_ptr(p.h, s)
                got = torch.as_tensor(_Dev(ptr, (ny, pitch), "<f4"), device="cuda")[:, :nx]
                assert torch.equal(got, dev[s])
    finally:
        for p in ps:
            p.close()
