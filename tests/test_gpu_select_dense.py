"""Dense selections over more blocks than the one-CTA tail takes: blocks of more
runs than the two-warp labelling holds, alone and among sparse ones, against
the oracle, and their labelling spread over the chip."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import compare as C  # noqa: E402
from oracle import fitrig_oracle as O  # noqa: E402
from paper_2509_21754_gb300 import fitrig as F  # noqa: E402


def noise(nsnap, ny, nx, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(nsnap, ny, nx, device="cuda", generator=g)


# 4 x 8 x 9 blocks of ragged maps (500 x 567 tiles); `mixed`: dense in one part
# of the image, hardly anything in the other.  tau near 0 selects about 40% of
# the tiles: some 900 runs a block (of a mixed image nearly all of the dense part,
# in few components, and 1.0 and 2.0 give many)
@pytest.mark.parametrize("tau", [0.01, 0.3, 1.0, 2.0])
@pytest.mark.parametrize("mixed", [False, True])
def test_many_dense_blocks(tau, mixed):
    stack = noise(6, 1500, 1700, 5)
    if mixed:
        stack[:, :, 700:] *= 0.05
        stack[:, 400:500, :] *= 0.05
    res = F.detect_stack(stack, 3, tau, F.BRANCH_IMAGE)
    x = stack.cpu().numpy()
    det = O.detect(x, 3, tau, F.BRANCH_IMAGE, "meanstd")
    di, dfq = C.library_decisions(res, tau)
    errs = C.compare(res["candidates"], x, 3, tau, F.BRANCH_IMAGE, "meanstd", decide_image=di,
                     decide_freq=dfq, det=det)
    assert not errs, errs[:5]
    assert len(res["candidates"]) > (1000 if tau >= 1.0 or not mixed else 0)


def test_dense_selection_is_spread_over_the_chip():
    """14 maps of 205 x 205 tiles, 224 blocks: labelling all blocks in full takes
    about twice as long as labelling sparse ones, and 30 times or more where a few CTAs
    take them in turn."""
    stack = noise(16, 1024, 1024, 7)
    us = {}
    for tau in (0.3, 6.0):
        with F.Plan(1024, 1024, 16, 5, tau, F.BRANCH_IMAGE) as p:
            p.push_stack(stack)
            times = []
            for _ in range(12):
                F.fitrig_detect(p.h)
                times.append(F.fitrig_kernel_ms(p.h, 2) * 1e3)
            us[tau] = min(times)
    assert us[0.3] < 6.0 * us[6.0], us
