"""The split transform of composite lengths and the radix transform's passes:
eta and its bin against numpy's FP64 transform, within the worst-case rounding
of the FP32 sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402


# composite lengths on both sides of each change of form: odd and even factors
# and sub-lengths, a square of a prime, the four- and eight-tile forms, twice a
# prime, a prime (direct), and every number of radix passes
@pytest.mark.parametrize("n", [67, 69, 70, 258, 289, 300, 998, 1001, 1498, 1664, 1665, 2021, 2994,
                               4093, 4095, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("harmonics", [1, 8])
def test_transform_of_length(n, harmonics):
    T = 37                                   # not a multiple of the tiles of a block
    g = torch.Generator(device="cuda").manual_seed(n)
    cube = torch.randn(n, T + 3, device="cuda", generator=g).square() + 0.5
    cube[::9, 5] += 4.0
    cube[3, 7] = float("nan")
    eta = torch.empty(T, device="cuda")
    kb = torch.empty(T, dtype=torch.int32, device="cuda")
    F.fitrig_spectrum_map(cube, n, T, T + 3, harmonics, eta, kb)
    y = cube.cpu().numpy()[:, :T].astype(np.float64)
    mag = np.abs(np.fft.rfft(y - y.mean(0), axis=0))[1:]
    # a sum of n FP32 terms is off by at most n 2^-24 times their magnitudes;
    # the shortest form of any length sums in at least two levels
    tol = n * 2.0 ** -24 * np.abs(y - y.mean(0)).sum(0)
    best = np.full(T, -1.0)
    of = np.zeros((mag.shape[0] + 1, T))     # the largest sum of each fundamental
    m = 1
    while m <= harmonics and m <= mag.shape[0]:
        k = np.arange(1, mag.shape[0] // m + 1)
        s = sum(mag[j * k - 1] for j in range(1, m + 1)) / np.sqrt(m)
        of[k] = np.maximum(of[k], s)
        best = np.maximum(best, s.max(0))
        m *= 2
    got, bins = eta.cpu().numpy(), kb.cpu().numpy()
    assert np.isnan(got[7]) and bins[7] == -1
    ok = np.arange(T) != 7
    assert (np.abs(got - best)[ok] <= tol[ok] * np.sqrt(harmonics)).all()
    assert (of[bins[ok], np.arange(T)[ok]] >= (best - 2 * tol * np.sqrt(harmonics))[ok]).all()
    assert (np.abs(got - best)[ok] / best[ok]).max() < 2e-6 * np.sqrt(n)
