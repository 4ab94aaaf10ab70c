"""Median/MAD of plans whose maps are larger than 2 Mi values: the split form
with its gather kernel on lent scratch, and its fallbacks (the cluster form up
to 8 Mi values, the grid-wide passes above), bit for bit against the
definition evaluated by sorting the library's own values in NumPy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402

MAD_TO_SIGMA = 1.482602218505602
# just above 2 Mi and 8 Mi values, neither a multiple of the pass's chunk
SIZES = [(1449, 1451), (2900, 2901)]


def definition(v: np.ndarray):
    v = v[np.isfinite(v)]
    k = (v.size - 1) // 2
    med = np.partition(v, k)[k]
    return float(med), MAD_TO_SIGMA * float(np.partition(np.abs(v - med), k)[k])


def values(kind: str, n: int):
    g = torch.Generator(device="cuda").manual_seed(n % 1009)
    v = torch.randn(n, device="cuda", generator=g).abs() + 0.1
    if kind == "quantised":              # ties in every bin
        v = (v * 8).round() / 8
    elif kind == "half_zero":            # the median's bracket overflows its chunks
        v[: n // 2 + n // 8] = 0.0
    elif kind == "nan":
        v[::97] = float("nan")
    elif kind == "sorted":               # a chunk holds only neighbours in value
        v = v.sort().values
    return v


@pytest.mark.parametrize("ny,nx", SIZES)
@pytest.mark.parametrize("kind", ["skewed", "quantised", "half_zero", "nan", "sorted"])
def test_large_map_noise_equals_definition(ny, nx, kind):
    # 1 x 1 tiles with x0 = x1 = 0: Delta = |x2| and r = 1, so v = x2^2
    stack = torch.zeros(3, ny, nx, device="cuda")
    stack[2] = values(kind, ny * nx).view(ny, nx)
    res = F.detect_stack(stack, 1, 50.0, F.BRANCH_IMAGE, noise=F.NOISE_MEDMAD)
    assert tuple(res["noise"][0]) == definition(res["values"][0].ravel())


@pytest.mark.parametrize("max_selected", [0, 1000])
def test_large_maps_of_both_branches(max_selected):
    """Three units and eta in one detect; with a selection limit too small to
    lend the scratch, the multi-pass form gives the same estimates."""
    ny, nx = SIZES[1]
    g = torch.Generator(device="cuda").manual_seed(5)
    stack = torch.randn(5, ny, nx, device="cuda", generator=g)
    with F.Plan(nx, ny, 5, 1, 1e6, F.BRANCH_BOTH, noise=F.NOISE_MEDMAD,
                max_selected=max_selected) as p:
        p.push_stack(stack)
        F.fitrig_detect(p.h)
        F.fitrig_detect(p.h)
        for s in range(3):
            assert F.fitrig_noise_params(p.h, s) == definition(F.fitrig_unit_values(p.h, s).ravel())
        assert F.fitrig_noise_params(p.h, -1) == definition(F.fitrig_spectrum(p.h)[0].ravel())
