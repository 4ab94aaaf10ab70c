"""The stack march where its form changes: a thread per tile at windows 1 and 2,
columns at 7 and 9 to 15, time segments for small images of long series, running
maxima over more than 16 snapshots; and the median/MAD of maps at the limit of
the resident form.  Against the oracle at its 1e-5 on tile values (a value is a
handful of FP32 operations on exact inputs), order statistics bit for bit."""
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

TYPES = {"f32": (F.F32, torch.float32), "bf16": (F.BF16, torch.bfloat16),
         "f16": (F.F16, torch.float16)}
MAD_TO_SIGMA = 1.482602218505602


def check(L, ny, nx, w, storage="f32", signed=False, running=False, branch=F.BRANCH_IMAGE):
    st, tdt = TYPES[storage]
    spec = synth.small_spec(L, ny, nx, n_steady=4, n_pulsed=2, pulse_period=(3, 4))
    stack, _ = synth.make_stack(spec, seed=31 * w + L + nx, device="cuda")
    if running:
        stack[:, ny // 2, nx // 3] = torch.linspace(100.0, 700.0, L, device="cuda")
    tau = 3.0
    rmode, mmode = ("signed" if signed else "abs"), ("running" if running else "global")
    res = F.detect_stack(stack, w, tau, branch, st,
                         rmode=F.RMODE_SIGNED if signed else F.RMODE_ABS,
                         mmode=F.MMODE_RUNNING if running else F.MMODE_GLOBAL)
    x = stack.to(tdt).float().cpu().numpy()
    det = O.detect(x, w, tau, branch, "meanstd", rmode, mmode=mmode)
    ok, worst = C.values_close(res["values"], np.stack([u.numerator for u in det.units]), rel=1e-5)
    assert ok, worst
    assert res["M"] == det.M and list(res["M_units"]) == list(det.M_units)
    di, dfq = C.library_decisions(res, tau)
    errs = C.compare(res["candidates"], x, w, tau, branch, "meanstd", rmode, "partial", di, dfq, det)
    assert not errs, errs[:5]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("signed", [False, True])
@pytest.mark.parametrize("w", [1, 2, 7, 9, 10, 11, 12, 13, 14, 15])
def test_windows_on_ragged_images(w, signed, storage):
    check(5, max(4 * w + 3, 11), 9 * w + 131, w, storage, signed)


@pytest.mark.parametrize("w", [1, 5, 8, 12, 16])
@pytest.mark.parametrize("running", [False, True])
def test_segments_of_a_long_series(w, running):
    check(99, 41, 83, w, running=running, branch=F.BRANCH_BOTH)


@pytest.mark.parametrize("n", [1, 2, 2049, 48 * 1024 - 1, 48 * 1024, 48 * 1024 + 1, 300_000, 1 << 21])
@pytest.mark.parametrize("kind", ["skewed", "constant", "nan"])
def test_noise_at_the_resident_limit(n, kind):
    groups = 3
    g = torch.Generator(device="cuda").manual_seed(n)
    v = torch.randn(groups, n, device="cuda", generator=g).square()
    if kind == "constant":
        v[:] = 0.75
    elif kind == "nan":
        v[:, 5::7] = float("nan")
    out = torch.zeros(2 * groups, dtype=torch.float64, device="cuda")
    assert F.fitrig_noise_static(v, groups, n, F.NOISE_MEDMAD, out) == F.OK
    torch.cuda.synchronize()
    for k in range(groups):
        x = v[k].cpu().numpy()
        x = x[np.isfinite(x)]
        med = np.sort(x)[(x.size - 1) // 2]
        mad = np.sort(np.abs(x - med))[(x.size - 1) // 2]
        assert out[2 * k].item() == float(med)
        assert out[2 * k + 1].item() == MAD_TO_SIGMA * float(mad)
