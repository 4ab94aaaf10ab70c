"""The sliding march's ratio r = min(Delta / |x|, 1) where the reference pixel x
is subnormal: the approximate reciprocal is infinite there, so such pixels take
the division, whatever the window."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import torch.nn.functional as tf  # noqa: E402

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402


# wide enough that warps lie inside the image, where the pixels decide the form
@pytest.mark.parametrize("w", [1, 3, 5, 7, 9, 11])
@pytest.mark.parametrize("scale", [1e-38, 1e-39])
def test_subnormal_reference_pixels(w, scale):
    ny, nx = 61, 419
    rng = np.random.default_rng(w)
    x = (scale * (1 + 0.3 * rng.random((3, ny, nx)))).astype(np.float32)
    x[:, ::3, ::3] = np.array([1.0, 2.0, 4.0], np.float32)[:, None, None]   # v does not underflow
    with F.Plan(nx, ny, 3, w, 6.0, F.BRANCH_IMAGE, stride=F.STRIDE_SLIDING) as p:
        p.push_stack(torch.from_numpy(x).cuda())
        F.fitrig_detect(p.h)
        got = F.fitrig_unit_values(p.h, 0).reshape(ny, nx).astype(np.float64)
    a = torch.from_numpy(x.astype(np.float64))
    delta = ((a[2] - a[1]).abs() - (a[1] - a[0]).abs()).abs()
    ratio = (delta / a[1].abs()).clamp(max=1.0)

    def mean(q):
        return tf.avg_pool2d(q[None], w, 1, w // 2, count_include_pad=False)[0]

    want = (mean(delta) * tf.max_pool2d(delta[None], w, 1, w // 2)[0] * mean(ratio)).numpy()
    seen = want > 1e-30   # a window of subnormal pixels alone underflows
    assert seen.sum() >= ny * nx // 9
    # sums of 2 w terms in a row, the ratio's two roundings, the product's four
    np.testing.assert_allclose(got[seen], want[seen], rtol=(4 * w + 8) * 2.0 ** -24, atol=0)
