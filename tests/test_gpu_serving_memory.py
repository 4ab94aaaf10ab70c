"""A serving field reserves what its trigger uses: maps of up to 48 Ki tiles take
the median/MAD in shared memory, without the scratch of larger maps."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402


def reserved(side, noise, freq):
    srv = F.fitrig_server_create(8 << 30, 1)
    try:
        if freq:
            rc, _ = F.fitrig_server_admit_freq(srv, side, side, 5, 6.0, F.BF16, noise, 8)
        else:
            rc, _ = F.fitrig_server_admit(srv, side, side, 5, 6.0, F.BF16, noise)
        assert rc == F.OK
        return F.fitrig_server_usage(srv)[0]
    finally:
        F.fitrig_server_destroy(srv)


# 100 x 100 and 221 x 221 tiles; 222 x 222 is above 48 Ki
@pytest.mark.parametrize("side,small", [(500, True), (1105, True), (1110, False)])
@pytest.mark.parametrize("freq", [False, True])
def test_small_maps_reserve_no_median_scratch(side, small, freq):
    extra = reserved(side, F.NOISE_MEDMAD, freq) - reserved(side, F.NOISE_MEANSTD, freq)
    assert extra == 0 if small else extra > 0
