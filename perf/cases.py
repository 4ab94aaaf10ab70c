"""The workloads the trigger's speed is judged on, through the library's public calls.

A case is a dict of plain values; ``kind`` says which call it stands for:

``detect``    a plan whose snapshots are resident: one detect and its candidates
              (with ``maps`` the eta map too), as a pipeline runs it that images
              straight into the plan's stack;
``stack``     a plan that is kept while stacks come and go: reset, push of a whole
              stack (from device or pinned host memory), detect, candidates;
``batch``     many fields of uneven size and snapshot count in one batch;
``serve``     fields that stream snapshots through a server: one snapshot each;
``spectrum``  the frequency statistic alone on a cube of tile series;
``noise``     the allocation-free noise estimate of a set of maps.

Inputs are the synthetic dirty-image stacks of the package (beam, correlated
noise, steady and pulsed sources), seeded.
"""
import math
import random

import numpy as np
import torch
import torch.nn.functional as tf

from paper_2509_21754_gb300 import fitrig as F
from paper_2509_21754_gb300 import synth

STORAGE = {"f32": F.F32, "bf16": F.BF16, "f16": F.F16}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BRANCH = {"image": F.BRANCH_IMAGE, "freq": F.BRANCH_FREQ, "both": F.BRANCH_BOTH}
NOISE = {"meanstd": F.NOISE_MEANSTD, "medmad": F.NOISE_MEDMAD}
GUARD = float(np.float32(1e-6))          # x-hat where x = 0 (Eq. 5)
MAD_TO_SIGMA = 1.482602218505602


def _case(name, kind, **kw):
    return dict({"name": name, "kind": kind}, **kw)


def _field(nsnap, ny, nx, window=5, storage="f32", branch="both", noise="medmad", nsigma=6.0,
           coding="value", sliding=False, signed=False, running=False, drop=False, harmonics=1,
           maps=False):
    return dict(nsnap=nsnap, ny=ny, nx=nx, window=window, storage=storage, branch=branch,
                noise=noise, nsigma=nsigma, coding=coding, sliding=sliding, signed=signed,
                running=running, drop=drop, harmonics=harmonics, maps=maps)


def listed():
    return [
        # the plain image-domain trigger on a small cut-out, stack after stack: latency counts
        _case("small_stack", "stack", source="device",
              **_field(16, 512, 512, branch="image", noise="meanstd")),
        # the main workload: 64 snapshots of 4096 x 4096, both branches, robust noise
        _case("main_field", "detect", **_field(64, 4096, 4096)),
        # the same field in difference-coded half storage
        _case("coded_field", "detect", **_field(64, 4096, 4096, storage="bf16", coding="delta")),
        # a window centred on every pixel, for positions finer than a tile
        _case("sliding_field", "detect", **_field(32, 4096, 4096, branch="image", sliding=True)),
        # a wide field: few snapshots, maps of tens of millions of tiles
        _case("wide_field", "detect", **_field(8, 24576, 24576)),
        # an hour's long series at window 32, frequency branch with harmonic summing
        _case("long_series", "detect", **_field(1500, 2048, 2048, window=32, branch="freq",
                                                noise="meanstd", harmonics=8, maps=True)),
        # an odd-sized field, a window without a special march, signed ratio, running M
        _case("odd_window", "detect", **_field(24, 3001, 2777, window=12, storage="f16",
                                               noise="meanstd", nsigma=5.0, signed=True,
                                               running=True, drop=True, maps=True)),
        # stacks that arrive from the host, rows that do not fill the device pitch
        _case("host_stack", "stack", source="host", **_field(20, 2600, 3100, storage="bf16", maps=True)),
        # a survey's fields of uneven size in one batch
        _case("field_batch", "batch", fields=16, lo=1024, hi=4096, snap_lo=16, snap_hi=40, mix=11),
        # fields that stream snapshots in real time
        _case("serving_round", "serve", fields=8, lo=1024, hi=5120, mix=7, noise="medmad",
              nsigma=12.0),
        # the transform alone: a cube of long series
        _case("series_cube", "spectrum", n=1024, T=16384, harmonics=1),
        # the noise estimate of a real-time loop that may not allocate
        _case("noise_maps", "noise", groups=62, n=672400, noise="medmad"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["detect", "detect", "detect", "sliding", "stack", "batch", "serve",
                       "spectrum", "noise"])
    if kind == "batch":
        lo = _log(rng, 300, 2000)
        return dict(kind="batch", fields=rng.randint(3, 16), lo=lo, hi=_log(rng, lo + 50, 4096),
                    snap_lo=rng.randint(5, 16), snap_hi=rng.randint(17, 48), mix=rng.randint(0, 999))
    if kind == "serve":
        lo = _log(rng, 400, 2000)
        return dict(kind="serve", fields=rng.randint(2, 16), lo=lo, hi=_log(rng, lo + 50, 5120),
                    mix=rng.randint(0, 999), noise=rng.choice(["medmad", "meanstd"]), nsigma=12.0)
    if kind == "spectrum":
        n = rng.choice([_log(rng, 8, 4096), 2 * _log(rng, 8, 2000), 2 ** rng.randint(7, 12)])
        return dict(kind="spectrum", n=n, T=_log(rng, 500, min(60000, 30_000_000 // n)),
                    harmonics=rng.choice([1, 1, 8]))
    if kind == "noise":
        groups = _log(rng, 1, 64)
        return dict(kind="noise", groups=groups, n=_log(rng, 3000, min(8_000_000, 40_000_000 // groups)),
                    noise=rng.choice(["medmad", "medmad", "meanstd"]))
    sliding = kind == "sliding"
    pixels = math.exp(rng.uniform(math.log(2.0 ** 17), math.log(2.0e7 if sliding or kind == "stack" else 4.0e8)))
    aspect = math.exp(rng.uniform(-0.5, 0.5))
    ny, nx = int(math.sqrt(pixels / aspect)), int(math.sqrt(pixels * aspect))
    most = (3.0e8 if sliding or kind == "stack" else 1.0e9) / pixels
    nsnap = _log(rng, 4, max(5, min(1500, most)))
    storage = rng.choice(["f32", "f32", "bf16", "f16"])
    if sliding:
        f = _field(nsnap, ny, nx, window=rng.choice([3, 5, 5, 7, 9, 11]), branch="image",
                   storage=storage, noise=rng.choice(["medmad", "meanstd"]), sliding=True)
        return dict(kind="detect", **f)
    window = rng.choice([5, 5, 5, 3, 4, 6, 8, 16, 32, 7, 12])
    coded = storage != "f32" and window in (3, 4, 5, 6, 8, 16, 32) and rng.random() < 0.5
    f = _field(nsnap, ny, nx, window=window, storage=storage,
               branch=rng.choice(["image", "both", "both", "freq"]),
               noise=rng.choice(["medmad", "medmad", "meanstd"]),
               coding="delta" if coded and kind == "detect" else "value",
               signed=rng.random() < 0.15, running=rng.random() < 0.25, drop=rng.random() < 0.2,
               harmonics=rng.choice([1, 1, 8]))
    if kind == "stack":
        return dict(kind="stack", source=rng.choice(["device", "device", "host"]), **f)
    return dict(kind="detect", **f)


# ---------------------------------------------------------------- inputs
def _snapshots(case, seed):
    """One FP32 snapshot after another, as the field's imager delivers them."""
    spec = synth.small_spec(case["nsnap"], case["ny"], case["nx"])
    for _, snap in synth.iter_stack(spec, seed, "cuda"):
        yield snap


def _mix_fields(case):
    """(snapshots, side) of a batch's or a server's fields."""
    rng = random.Random(case["mix"])
    lo, hi = case.get("snap_lo", 3), case.get("snap_hi", 3)
    return [(rng.randint(lo, hi), rng.randint(case["lo"], case["hi"])) for _ in range(case["fields"])]


def _batch_field(nsnap, side):
    return _field(nsnap, side, side, storage="bf16")


def _batch_snapshots(nsnap, side, seed):
    for _, snap in synth.iter_stack(synth.batched_spec(nsnap, side), seed, "cuda"):
        yield snap


def _series(case, seed):
    """Tile series as the march leaves them: skewed, with pulses in a few of them."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, T = case["n"], case["T"]
    cube = torch.randn(n, T, generator=g, device="cuda").square_().add_(0.5)
    pulsed = torch.randint(0, T, (max(1, T // 50),), generator=g, device="cuda")
    cube[seed % 3::7, pulsed] += 6.0
    return cube


def _maps(case, seed):
    """Maps of the tile statistic: positive, right-skewed, a few invalid tiles."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(case["groups"], case["n"], generator=g, device="cuda").abs_().mul_(3.0).add_(0.5)
    v *= torch.rand(case["groups"], case["n"], generator=g, device="cuda").add_(0.2)
    v[:, seed % 97::5003] = float("nan")
    return v


def _pinned_candidates(count):
    return torch.zeros(count, 8, dtype=torch.int32, pin_memory=True).numpy().view(F.CANDIDATE_DTYPE)[:, 0]


class _State:
    """A prepared case; frees the library's handles when it goes."""

    def __init__(self, case):
        self.case = case
        self.plans, self.batch, self.server = [], None, None

    def __del__(self):
        if self.batch is not None:
            F.fitrig_batch_destroy(self.batch)
        if self.server is not None:
            F.fitrig_server_destroy(self.server)
        for p in self.plans:
            p.close()


def _plan(f, autotune=False):
    return F.Plan(f["nx"], f["ny"], f["nsnap"], f["window"], f["nsigma"], BRANCH[f["branch"]],
                  STORAGE[f["storage"]], NOISE[f["noise"]],
                  rmode=F.RMODE_SIGNED if f["signed"] else F.RMODE_ABS,
                  edge=F.EDGE_DROP if f["drop"] else F.EDGE_PARTIAL,
                  stride=F.STRIDE_SLIDING if f["sliding"] else F.STRIDE_TILE, autotune=autotune,
                  mmode=F.MMODE_RUNNING if f["running"] else F.MMODE_GLOBAL,
                  harmonics=f["harmonics"],
                  coding=F.CODING_DELTA if f["coding"] == "delta" else F.CODING_VALUE)


def _room(f):
    """Candidates that the caller's buffer has room for."""
    tiles = f["ny"] * f["nx"] // (5 if f["sliding"] else f["window"] ** 2)
    return 4096 + (1 if f["branch"] == "freq" else f["nsnap"] - 2) * tiles // 12


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind in ("detect", "stack"):
        s.plans = [_plan(case)]
        s.out = [_pinned_candidates(_room(case))]
        if kind == "detect":
            for snap in _snapshots(case, seed):
                F.fitrig_push_snapshot(s.plans[0].h, snap)
        else:
            shape = (case["nsnap"], case["ny"], case["nx"])
            dtype = DTYPE[case["storage"]]
            if case["source"] == "host":
                s.block = torch.empty(shape, dtype=dtype, pin_memory=True)
            else:
                s.block = torch.empty(shape, dtype=dtype, device="cuda")
            for k, snap in enumerate(_snapshots(case, seed)):
                s.block[k].copy_(snap.to(dtype))
    elif kind == "batch":
        for k, (nsnap, side) in enumerate(_mix_fields(case)):
            p = _plan(_batch_field(nsnap, side), autotune=True)
            s.plans.append(p)
            for snap in _batch_snapshots(nsnap, side, seed * 100 + k):
                F.fitrig_push_snapshot(p.h, snap)
        s.out = [_pinned_candidates(_room(_batch_field(*f))) for f in _mix_fields(case)]
        s.batch = F.fitrig_batch_create(s.plans)
    elif kind == "serve":
        s.server = F.fitrig_server_create(64 << 30, case["fields"])
        s.pools, s.next = [], 2
        s.out = [np.zeros(_SERVED, F.CANDIDATE_DTYPE) for _ in range(case["fields"])]
        s.count = [0] * case["fields"]
        for k, (_, side) in enumerate(_mix_fields(case)):
            pool = torch.empty(3, side, side, dtype=torch.bfloat16, pin_memory=True)
            for j, snap in enumerate(_batch_snapshots(3, side, seed * 100 + k)):
                pool[j].copy_(snap.to(torch.bfloat16))
            s.pools.append(pool)
            F.fitrig_server_admit(s.server, side, side, 5, case["nsigma"], F.BF16,
                                  NOISE[case["noise"]])
            for j in range(2):
                F.fitrig_server_push(s.server, k, pool[j], 0)
        F.fitrig_server_drain(s.server)
    elif kind == "spectrum":
        s.cube = _series(case, seed)
        s.eta = torch.empty(case["T"], device="cuda")
        s.bin = torch.empty(case["T"], dtype=torch.int32, device="cuda")
    else:
        s.maps = _maps(case, seed)
        s.cs = torch.empty(2 * case["groups"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return s


# ---------------------------------------------------------------- one pass
_SERVED = 65536   # candidates that a served unit delivers at most


def _candidates(s, k, n):
    """The last detect's candidates in the caller's buffer (its rest stays zero) and their number."""
    F.fitrig_candidates(s.plans[k].h, out=s.out[k])
    return dict({c: s.out[k][c] for c in F.CANDIDATE_DTYPE.names}, count=int(n))


def run(state):
    s, case = state, state.case
    kind = case["kind"]
    if kind in ("detect", "stack"):
        h = s.plans[0].h
        if kind == "stack":
            F.fitrig_plan_reset(h)
            F.fitrig_push_snapshots(h, s.block)
        _, n = F.fitrig_detect(h)
        got = _candidates(s, 0, n)
        if case["maps"]:
            got["eta"], got["bin"] = F.fitrig_spectrum(h)
        return got
    if kind == "batch":
        _, n = F.fitrig_batch_detect(s.batch, len(s.plans))
        got = [_candidates(s, k, n[k]) for k in range(len(s.plans))]
        return [n] + [[c["x"], c["y"], c["significance"]] for c in got]
    if kind == "serve":
        for k, pool in enumerate(s.pools):
            F.fitrig_server_push(s.server, k, pool[s.next], 0)
        s.next = (s.next + 1) % 3
        F.fitrig_server_drain(s.server)
        res, cands = F.fitrig_server_poll(s.server)
        status = [0] * len(s.pools)
        for r in res:
            k, n = r["field"], int(r["ncand"])
            s.out[k][:n] = cands[r["cand_offset"]:r["cand_offset"] + n]
            s.out[k][n:s.count[k]] = 0
            s.count[k], status[k] = n, int(r["status"])
        return {"status": np.array(status), "count": np.array(s.count),
                "fields": [(c["x"], c["y"], c["significance"]) for c in s.out]}
    if kind == "spectrum":
        F.fitrig_spectrum_map(s.cube, case["n"], case["T"], case["T"], case["harmonics"], s.eta, s.bin)
        return {"eta": s.eta, "bin": s.bin}
    F.fitrig_noise_static(s.maps, case["groups"], case["n"], NOISE[case["noise"]], s.cs)
    return s.cs


def work(case):
    kind = case["kind"]
    if kind in ("detect", "stack"):
        px = case["nsnap"] * case["ny"] * case["nx"]
        flops = 10.0 * px * (case["window"] if case["sliding"] else 1)
        return {"bytes": px * (4 if case["storage"] == "f32" else 2), "flops": flops}
    if kind == "batch":
        px = sum(n * side * side for n, side in _mix_fields(case))
        return {"bytes": 2 * px, "flops": 10.0 * px}
    if kind == "serve":   # the unit's three snapshots, one of them new
        px = 3 * sum(side * side for _, side in _mix_fields(case))
        return {"bytes": 2 * px, "flops": 10.0 * px}
    if kind == "spectrum":
        n, T = case["n"], case["T"]
        return {"bytes": 4 * n * T + 8 * T, "flops": 2.5 * n * math.log2(n) * T}
    return {"bytes": 4 * case["groups"] * case["n"], "flops": 4.0 * case["groups"] * case["n"]}


# ---------------------------------------------------------------- the same in 64 bits
def _stored(case, snaps):
    """The snapshots as the plan stores (and, difference-coded, decodes) them."""
    half = DTYPE[case["storage"]]
    last = None
    for snap in snaps:
        if case["storage"] == "f32":
            yield snap
        elif case["coding"] == "delta":
            last = snap if last is None else last + (snap - last).to(half).float()
            yield last
        else:
            yield snap.to(half).float()


def _tile_sum(x, w):
    ny, nx = x.shape
    x = tf.pad(x, (0, -nx % w, 0, -ny % w))
    return x.view(x.shape[0] // w, w, x.shape[1] // w, w).sum((1, 3))


def _statistic(case, a, b, c):
    """v of one unit from its three snapshots."""
    w = case["window"]
    d = ((c - b).abs() - (b - a).abs()).abs()
    ref = b if case["signed"] else b.abs()
    r = (d / torch.where(b == 0, GUARD, ref)).clamp(max=1.0)
    one = torch.ones_like(d)
    if case["sliding"]:
        def total(x):
            return tf.avg_pool2d(x[None, None], w, 1, w // 2, divisor_override=1)[0, 0]
        top = tf.max_pool2d(d[None, None], w, 1, w // 2)[0, 0]
    else:
        def total(x):
            return _tile_sum(x, w)
        ny, nx = d.shape
        top = tf.max_pool2d(tf.pad(d, (0, -nx % w, 0, -ny % w))[None, None], w, w)[0, 0]
    n = total(one)
    return total(d) / n * top * (total(r) / n)


def _spread(v, noise):
    v = v.reshape(-1)
    if noise == "meanstd":
        return v.mean(), v.std(unbiased=False)
    k = (v.numel() - 1) // 2
    mid = v.sort().values[k]
    return mid, MAD_TO_SIGMA * (v - mid).abs().sort().values[k]


def _peaks(z, tau):
    """Tiles that are the largest of their 8-connected component of z > tau."""
    low = torch.full_like(z, -math.inf)
    best = torch.where(z > tau, z, low)
    while True:
        was = best
        for _ in range(8):
            best = torch.where(z > tau, tf.max_pool2d(best[None, None], 3, 1, 1)[0, 0], low)
        if torch.equal(was, best):
            break
    ty, tx = torch.where((z > tau) & (z == best))
    return ty, tx


def _exact_detect(case, snaps, room):
    """The candidates' floating values; where a field has so many tiles that some lie within
    FP32 rounding of the threshold, the lists need not line up, and there is no such value."""
    w = 1 if case["sliding"] else case["window"]
    ny, nx = case["ny"], case["nx"]
    if case["drop"]:
        ny, nx = ny // w * w, nx // w * w
    units = 1 if case["branch"] == "freq" else case["nsnap"] - 2
    lists = units * ny * nx <= 1_500_000 * w * w
    image, series, biggest, last = [], [], [], []
    for snap in _stored(case, snaps):
        last.append(snap[:ny, :nx].double())
        biggest.append(last[-1].max())
        if len(last) < 3:
            continue
        a, b, c = last
        v = _statistic(case, a, b, c)
        if case["branch"] != "image":
            series.append(v)
        if case["branch"] != "freq" and lists:
            centre, scale = _spread(v, case["noise"])
            z = (v - centre) / scale
            ty, tx = _peaks(z, case["nsigma"])
            i = torch.arange(w * w, device=v.device)
            y = (ty[:, None] * w + i // w).clamp(max=ny - 1)
            x = (tx[:, None] * w + i % w).clamp(max=nx - 1)
            at = y * nx + x
            a1, b1, c1 = (q.reshape(-1)[at] for q in (a, b, c))
            d = ((c1 - b1).abs() - (b1 - a1).abs()).abs()
            j = torch.where(d == d.max(1, keepdim=True).values, i, w * w).min(1, keepdim=True).values
            at, order = at.gather(1, j)[:, 0].sort()
            image.append((z[ty, tx][order], (at % nx).double(), (at // nx).double()))
        del last[0]
    found, eta = [], None
    if case["branch"] != "image" and (lists or case["maps"]):
        z, xf, yf, eta = _exact_freq(case, series, biggest, ny, nx)
        found.append((z, xf, yf))
    found += image
    got = dict({k: None for k in F.CANDIDATE_DTYPE.names}, count=None)
    if lists:
        z, x, y = (torch.cat(q).float() for q in zip(*found))
        got.update({k: tf.pad(q[:room], (0, room - min(room, len(q))))
                    for k, q in (("significance", z), ("xf", x), ("yf", y))})
    if case["maps"]:
        got.update(eta=eta.float(), bin=None)
    return got if lists or case["maps"] else None


def _magnitudes(v, harmonics):
    """The largest (harmonic sum of) spectral magnitudes of series along dim 0."""
    mag = torch.fft.rfft(v - v.mean(0), dim=0)[1:].abs()
    best, m = mag.max(0).values, 2
    while m <= harmonics and m <= mag.shape[0]:
        k = torch.arange(1, mag.shape[0] // m + 1, device=v.device)
        best = torch.maximum(best, sum(mag[j * k - 1] for j in range(1, m + 1)).max(0).values / math.sqrt(m))
        m *= 2
    return best


def _exact_freq(case, series, biggest, ny, nx):
    w = case["window"]
    if case["running"]:
        top = torch.stack(biggest).cummax(0).values[2:].clamp(min=GUARD)
        series = [v * (top[-1] / m) ** 2 for v, m in zip(series, top)]
    shape = series[0].shape
    flat = [v.reshape(-1) for v in series]
    step = max(1, 100_000_000 // len(flat))
    eta = torch.cat([_magnitudes(torch.stack([v[k:k + step] for v in flat]), case["harmonics"])
                     for k in range(0, flat[0].numel(), step)]).reshape(shape)
    centre, scale = _spread(eta, case["noise"])
    z = (eta - centre) / scale
    ty, tx = _peaks(z, case["nsigma"])

    def vertex(dy, dx):
        pad = tf.pad(eta, (1, 1, 1, 1), value=math.nan)
        lo, mid, hi = pad[ty + 1 - dy, tx + 1 - dx], eta[ty, tx], pad[ty + 1 + dy, tx + 1 + dx]
        den = lo - 2 * mid + hi
        return torch.where(den < 0, 0.5 * (lo - hi) / den, 0.0).clamp(-0.5, 0.5)

    wide = (nx - tx * w).clamp(max=w)
    high = (ny - ty * w).clamp(max=w)
    xf = tx * w + 0.5 * (wide - 1) + vertex(0, 1) * w
    yf = ty * w + 0.5 * (high - 1) + vertex(1, 0) * w
    return z[ty, tx], xf, yf, eta.reshape(shape)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("detect", "stack"):
        return _exact_detect(case, _snapshots(case, seed), _room(case))
    if kind == "batch":
        got = []
        for k, (n, side) in enumerate(_mix_fields(case)):
            f = _batch_field(n, side)
            got.append(_exact_detect(f, _batch_snapshots(n, side, seed * 100 + k), _room(f)))
        return [None] + [c and [None, None, c["significance"]] for c in got] if any(got) else None
    if kind == "serve":
        got = []
        for k, (_, side) in enumerate(_mix_fields(case)):
            f = _field(3, side, side, storage="bf16", branch="image", noise=case["noise"],
                       nsigma=case["nsigma"])
            c = _exact_detect(f, _batch_snapshots(3, side, seed * 100 + k), _SERVED)
            got.append(c and (None, None, c["significance"]))
        return {"status": None, "count": None, "fields": got} if any(got) else None
    if kind == "spectrum":
        return {"eta": _magnitudes(_series(case, seed).double(), case["harmonics"]).float(), "bin": None}
    v = _maps(case, seed).double()
    return torch.stack([torch.stack(_spread(m[m.isfinite()], case["noise"])) for m in v]).reshape(-1)
