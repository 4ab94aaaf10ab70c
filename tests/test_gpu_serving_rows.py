"""Serving fields whose snapshots are large and whose rows do not fill the device
pitch (they are copied linearly and set at their pitch on the device): each
unit equals the batch trigger's, alone or pushed from several threads at once,
and the pushes take no device memory beside the fields' reservations."""
import threading
import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2509_21754_gb300 import fitrig as F  # noqa: E402
from paper_2509_21754_gb300 import synth  # noqa: E402

# pieces of a snapshot that the lent buffers take: one, one (pixels as tiles), four,
# and none (pitched copies)
FIELDS = [(1499, 1499, 5, F.BF16, torch.bfloat16, True),
          (1100, 1001, 1, F.F32, torch.float32, True),
          (2303, 2001, 8, F.F16, torch.float16, False),
          (1301, 1204, 16, F.F32, torch.float32, True)]
L = 6


def stacks():
    out = []
    for k, (ny, nx, _, _, dt, pinned) in enumerate(FIELDS):
        st, _ = synth.make_stack(synth.small_spec(L, ny, nx, n_pulsed=3, pulse_period=(3, 5)), seed=20 + k,
                                 device="cuda")
        h = st.to(dt).cpu()
        out.append(h.pin_memory() if pinned else h)
    torch.cuda.empty_cache()
    return out


def test_units_from_several_threads_equal_the_batch_trigger():
    data = stacks()
    want = []
    for x, (_, _, w, storage, _, _) in zip(data, FIELDS):
        ref = F.detect_stack(x.cuda(), w, 8.0, F.BRANCH_IMAGE, storage, F.NOISE_MEDMAD, dumps=False)
        want.append(ref["candidates"])
    torch.cuda.empty_cache()
    srv = F.fitrig_server_create(16 << 30, len(FIELDS))
    try:
        for ny, nx, w, storage, _, _ in FIELDS:
            rc, _ = F.fitrig_server_admit(srv, nx, ny, w, 8.0, storage, F.NOISE_MEDMAD)
            assert rc == F.OK
        free = torch.cuda.mem_get_info()[0]

        def feed(ids):
            for k in range(L):
                for i in ids:
                    assert F.fitrig_server_push(srv, i, data[i][k], time.monotonic_ns()) == F.OK

        threads = [threading.Thread(target=feed, args=(ids,)) for ids in ([0, 2], [1, 3])]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        F.fitrig_server_drain(srv)
        assert free - torch.cuda.mem_get_info()[0] < 16 << 20   # (what launches need; no buffers)
        res, cands = F.fitrig_server_poll(srv)
        assert len(res) == (L - 2) * len(FIELDS)
        for r in res:
            c = cands[r["cand_offset"]:r["cand_offset"] + r["ncand"]]
            ref = want[r["field"]]
            assert c.tobytes() == ref[ref["snapshot"] == r["unit"]].tobytes(), (r["field"], r["unit"])
            assert 0.0 <= r["copy_ms"] < 1e3
    finally:
        F.fitrig_server_destroy(srv)
