"""Components and candidate emission where their forms change: blocks with more
runs than the two-warp labelling holds, tile rows of more than 32 bitmap words,
and 1 x 1 tiles (sliding mode, windows of 1), against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import compare as C  # noqa: E402
from oracle import fitrig_oracle as O  # noqa: E402
from paper_2509_21754_gb300 import fitrig as F  # noqa: E402
from paper_2509_21754_gb300 import synth  # noqa: E402


def check(stack, w, tau, sliding=False, branch=F.BRANCH_BOTH):
    res = F.detect_stack(stack, w, tau, branch,
                         stride=F.STRIDE_SLIDING if sliding else F.STRIDE_TILE)
    x = stack.cpu().numpy()
    det = O.detect(x, w, tau, branch, "meanstd", stride="sliding" if sliding else "tile")
    di, dfq = C.library_decisions(res, tau)
    errs = C.compare(res["candidates"], x, 1 if sliding else w, tau, branch, "meanstd",
                     decide_image=di, decide_freq=dfq, det=det)
    assert not errs, errs[:5]
    return res


# tau near 0 selects about 40% of the tiles: some 900 runs in a 64 x 64 block
@pytest.mark.parametrize("tau", [0.01, 0.3, 6.0])
@pytest.mark.parametrize("ny,nx", [(192, 192), (203, 391)])
def test_blocks_of_many_runs(tau, ny, nx):
    g = torch.Generator(device="cuda").manual_seed(ny)
    check(torch.randn(4, ny, nx, device="cuda", generator=g), 3, tau)


@pytest.mark.parametrize("w,nx", [(3, 3 * 1024), (3, 3 * 1024 + 1), (4, 4 * 1100), (8, 8 * 1030 + 3)])
def test_rows_of_more_than_1024_tiles(w, nx):
    stack, _ = synth.make_stack(synth.small_spec(4, 6 * w + 1, nx), seed=nx, device="cuda")
    assert len(check(stack, w, 2.0)["candidates"])


@pytest.mark.parametrize("nx", [1024, 1025, 2100])
@pytest.mark.parametrize("w,sliding", [(1, False), (3, True)])
def test_pixels_as_tiles(nx, w, sliding):
    stack, _ = synth.make_stack(synth.small_spec(4, 21, nx), seed=nx + w, device="cuda")
    check(stack, w, 1.5, sliding)
