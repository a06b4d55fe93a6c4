"""The calls that the performance of this library is measured on.

Every case is one call (or one compress + decompress pair) through the public
Python API, on inputs resident on the GPU, over the detector shapes, batch sizes
and options that the benchmark, the serving loop and the tests use.  A case is a
flat dict:

  op       "compress", "decompress", "roundtrip" or "static" (compress_frame_static)
  P, H, W  panels, rows and columns of a frame;  n: frames in the call
  mean, sd background;  hot: share of pixels at 5,000;  lo, hi: spots per frame
  bin, eb, dims, roi_coder, chunk, max_peaks, dense: the options that differ
           from the defaults (dense: the fused kernel's hot-pixel variant)

Inputs are seeded synthetic frames made on the GPU with the distributions of
synthetic/frames.py: Gaussian background clamped at 0, hot pixels, and Gaussian
Bragg spots.
"""
from __future__ import annotations

import math

import torch

import paper_2206_11297_gb300 as rb

_STAMP = 7  # a spot is drawn over +-7 px
_HOT = 5000.0

_CSPAD = dict(P=32, H=185, W=388, mean=20.0, sd=5.0, hot=0.0, lo=20, hi=100)
_EPIX = dict(P=16, H=352, W=384, mean=30.0, sd=8.0, hot=0.01, lo=0, hi=300, max_peaks=8192)
_JUNGFRAU = dict(P=8, H=512, W=1024, mean=20.0, sd=5.0, hot=0.0, lo=0, hi=500)
_OPTIONS = dict(bin=2, eb=10.0, dims=2, roi_coder=0, chunk=1, max_peaks=2048, dense=False)


def _case(name, op, detector, n, **options):
    c = dict(op=op, n=n, **_OPTIONS)
    c.update(detector)
    c.update(options)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one event on its own: an online monitor's latency
        _case("compress_cspad_1", "compress", _CSPAD, 1, lo=50, hi=50),
        # one detector module through the call that needs no context
        _case("static_module_1", "static", dict(_CSPAD, P=1, H=352, W=384, lo=0, hi=10), 1),
        # one request of the serving loop (1 to 64 frames)
        _case("compress_cspad_33", "compress", _CSPAD, 33),
        # the benchmark's batch
        _case("compress_cspad_1000", "compress", _CSPAD, 1000),
        # hot-pixel frames, about 3,600 windows each, in the variant the autotuner picks for them
        _case("compress_epix_hot_100", "compress", _EPIX, 100, dense=True),
        # the same detector on a context as the serving loop makes it, with coded
        # windows and a code shared by ten frames (an archive's settings)
        _case("compress_epix_coded_30", "compress", _EPIX, 30, roi_coder=1, chunk=10),
        # large panels, many spots
        _case("compress_jungfrau_20", "compress", _JUNGFRAU, 20),
        # a detector whose panels are odd in both directions
        _case("compress_odd_24", "compress", dict(_CSPAD, P=7, H=255, W=301, lo=0, hi=60), 24),
        # the 3-D predictor of the quality search: compress, then decompress
        _case("roundtrip_stack_40", "roundtrip", _CSPAD, 40, dims=3),
        # random access to one stored event
        _case("decompress_cspad_1", "decompress", _CSPAD, 1, lo=50, hi=50),
        # reading a run back
        _case("decompress_cspad_400", "decompress", _CSPAD, 400),
        # reading hot-pixel frames back: long codes, many windows
        _case("decompress_epix_60", "decompress", _EPIX, 60),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["cspad", "cspad", "epix", "epix_coded", "jungfrau", "odd", "static", "roundtrip",
                       "decompress", "decompress"])
    if kind == "cspad":
        lo, eb = rng.choice([0, 20, 50]), rng.choice([1.0, 10.0, 10.0, 50.0])
        return _case(None, "compress", _CSPAD, _log_int(rng, 1, 300 if eb < 10.0 else 900), lo=lo,
                     hi=lo + rng.randrange(10, 120), eb=eb)
    if kind == "epix":
        return _case(None, "compress", _EPIX, _log_int(rng, 1, 100), eb=rng.choice([1.0, 10.0, 50.0]), dense=True)
    if kind == "epix_coded":
        return _case(None, "compress", _EPIX, _log_int(rng, 1, 30), roi_coder=1, chunk=rng.choice([1, 8, 64]))
    if kind == "jungfrau":
        return _case(None, "compress", _JUNGFRAU, _log_int(rng, 1, 120), hi=rng.randrange(20, 500))
    if kind in ("odd", "static"):
        # generic panels, most of them odd, from a small module to a 1-megapixel one
        b = rng.choice([1, 2, 2, 2, 3, 4])
        P, H, W = rng.randrange(1, 9), _log_int(rng, 60, 700), _log_int(rng, 60, 1100)
        det = dict(_CSPAD, P=P, H=H, W=W, lo=0, hi=rng.randrange(2, 80))
        if kind == "static":
            det["P"] = min(P, 2) if H * W < 300_000 else 1  # the call's fixed scratch holds about a million bins
            return _case(None, "static", det, 1, bin=max(b, 2))
        if b == 1:  # a frame holds at most 5.7 million bins
            det["P"] = P = min(P, 5_500_000 // (H * W))
        return _case(None, "compress", det, _log_int(rng, 1, max(1, 20_000_000 // (P * H * W))), bin=b)
    if kind == "roundtrip":
        return _case(None, "roundtrip", _CSPAD, _log_int(rng, 1, 40), dims=rng.choice([1, 3]))
    det, most = rng.choice([(_CSPAD, 400), (_EPIX, 60), (_JUNGFRAU, 100)])
    return _case(None, "decompress", det, _log_int(rng, 1, most), eb=rng.choice([1.0, 10.0, 10.0, 50.0]))


def _geometry(case):
    return case["P"], case["H"], case["W"]


def _make(case, seed):
    """float32 [n, P, H, W] frames, and each spot's (frame, panel, row, col)."""
    P, H, W = _geometry(case)
    n, px = case["n"], P * H * W
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    frames = torch.empty((n, P, H, W), dtype=torch.float32, device="cuda")
    spots = []
    step = max(1, 100_000_000 // px)
    d = torch.arange(-_STAMP, _STAMP + 1, device="cuda")
    for f0 in range(0, n, step):
        part = frames[f0:f0 + step]
        m = part.shape[0]
        part.normal_(case["mean"], case["sd"], generator=g).clamp_(min=0.0)
        if case["hot"] > 0:
            at = torch.randint(0, px, (m, int(round(case["hot"] * px))), generator=g, device="cuda")
            part.view(m, px).scatter_(1, at, _HOT)
        count = torch.randint(case["lo"], case["hi"] + 1, (m,), generator=g, device="cuda")
        frame = torch.repeat_interleave(torch.arange(m, device="cuda"), count)
        k = frame.numel()
        if k == 0:
            continue
        panel = torch.randint(0, P, (k,), generator=g, device="cuda")
        u = torch.rand((4, k), generator=g, device="cuda", dtype=torch.float64)
        cy, cx, amp, sig = u[0] * H, u[1] * W, 200.0 + 1800.0 * u[2], 1.0 + 0.5 * u[3]
        row, col = cy.long().clamp_(max=H - 1), cx.long().clamp_(max=W - 1)
        yy, xx = row[:, None] + d, col[:, None] + d
        ey = torch.exp(-(yy + 0.5 - cy[:, None]) ** 2 / (2 * sig[:, None] ** 2))
        ex = torch.exp(-(xx + 0.5 - cx[:, None]) ** 2 / (2 * sig[:, None] ** 2))
        # whole 1/64 counts, so that overlapping spots add up the same in any order
        stamp = torch.round(amp[:, None, None] * ey[:, :, None] * ex[:, None, :] * 64.0) / 64.0
        ok = ((yy >= 0) & (yy < H))[:, :, None] & ((xx >= 0) & (xx < W))[:, None, :]
        base = ((frame * P + panel) * H)[:, None, None]
        at = (base + yy[:, :, None].clamp(0, H - 1)) * W + xx[:, None, :].clamp(0, W - 1)
        light = torch.zeros(m * px, dtype=torch.float32, device="cuda")
        light.index_add_(0, at[ok], stamp[ok].float())
        part.view(-1).add_(light)
        spots.append(torch.stack([frame + f0, panel, row, col]))
    return frames, torch.cat(spots, 1) if spots else torch.zeros((4, 0), dtype=torch.long, device="cuda")


def _params(case):
    return rb.default_params(bin_h=case["bin"], bin_w=case["bin"], abs_eb=case["eb"], lorenzo_dims=case["dims"],
                             roi_coder=case["roi_coder"], chunk_frames=case["chunk"], max_peaks=case["max_peaks"])


def _stride(case):
    """Bytes per output slot: a quarter of the raw frame, or the worst case of the
    windows where those may outweigh the frame's background."""
    raw = 4 * case["P"] * case["H"] * case["W"]
    room = raw if case["hot"] > 0 else raw // 4
    if case["op"] == "static" or case["bin"] == 1:
        return rb.compress_bound(_geometry(case), _params(case))
    return (room + 400_000 + 15) // 16 * 16


def _wanted(case, spots, frames):
    """Windows to keep, as a program that knows its peaks gives them: the spots and,
    on hot-pixel detectors, 3,000 hot pixels of each frame.  (panel, row, col) u16 as
    int16 [n, max_peaks, 3] and int32 [n], and the same as long [4, total]."""
    P, H, W = _geometry(case)
    n = case["n"]
    if case["hot"] > 0:
        order = torch.argsort((frames.view(n, -1) < _HOT).to(torch.uint8), dim=1, stable=True)[:, :3000]
        f = torch.arange(n, device="cuda")[:, None].expand_as(order)
        hot = torch.stack([f, order // (H * W), order // W % H, order % W]).reshape(4, -1)
        spots = torch.cat([spots, hot], 1)
        spots = spots[:, torch.argsort(spots[0], stable=True)]
    count = torch.bincount(spots[0], minlength=n)
    first = torch.cumsum(count, 0) - count
    peaks = torch.zeros((n, case["max_peaks"], 3), dtype=torch.int16, device="cuda")
    rank = torch.arange(spots.shape[1], device="cuda") - first[spots[0]]
    peaks[spots[0], rank] = spots[1:].t().to(torch.int16)
    return peaks, count.to(torch.int32), spots


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.op, s.n = case["op"], case["n"]
    frames, spots = _make(case, seed)
    s.geometry, s.params, s.stride = _geometry(case), _params(case), _stride(case)
    s.out = torch.zeros((s.n, s.stride), dtype=torch.uint8, device="cuda")
    s.frame_bytes = torch.zeros(s.n, dtype=torch.int64, device="cuda")
    s.status = torch.zeros(s.n, dtype=torch.int32, device="cuda")
    if s.op == "static":
        s.frames = frames
        return s
    s.ctx = rb.Context(s.geometry, s.params, max_frames=s.n)
    if case["dense"]:
        s.ctx.set_fused_dense_peaks(True)
    if s.op == "compress":
        s.frames = frames
        return s
    peaks, npeaks, _ = _wanted(case, spots, frames)
    s.restored = torch.empty((s.n, *s.geometry), dtype=torch.float32, device="cuda")
    s.restored_status = torch.zeros(s.n, dtype=torch.int32, device="cuda")
    if s.op == "roundtrip":
        s.frames, s.peaks, s.npeaks = frames, peaks, npeaks
        s.offsets = torch.arange(s.n, dtype=torch.int64, device="cuda") * s.stride
        return s
    # decompress: the streams back to back, as a file of them is read
    s.ctx.compress(frames, out=s.out, out_stride=s.stride, peaks=peaks, npeaks=npeaks,
                   frame_bytes=s.frame_bytes, status=s.status)
    if bool((s.status != 0).any()):
        raise RuntimeError("a frame of the decompression input was not compressed")
    sizes = s.frame_bytes.tolist()
    s.data = torch.cat([s.out[k, :b] for k, b in enumerate(sizes)])
    s.offsets = torch.cumsum(s.frame_bytes, 0) - s.frame_bytes
    s.out = None
    return s


def run(s):
    if s.op == "static":
        rb.compress_frame_static(s.geometry, s.params, s.frames[0], s.out[0], s.frame_bytes, s.status)
        return s.out, s.frame_bytes, s.status
    if s.op == "compress":
        return s.ctx.compress(s.frames, out=s.out, out_stride=s.stride, frame_bytes=s.frame_bytes, status=s.status)
    if s.op == "roundtrip":
        s.ctx.compress(s.frames, out=s.out, out_stride=s.stride, peaks=s.peaks, npeaks=s.npeaks,
                       frame_bytes=s.frame_bytes, status=s.status)
        s.ctx.decompress(s.out.view(-1), s.offsets, s.n, out=s.restored, status=s.restored_status)
        return s.out, s.frame_bytes, s.status, s.restored, s.restored_status
    return s.ctx.decompress(s.data, s.offsets, s.n, out=s.restored, status=s.restored_status)


def _stream_bytes(case):
    """About what a frame's stream takes: its windows and its coded bins."""
    bins = case["P"] * -(-case["H"] // case["bin"]) * -(-case["W"] // case["bin"])
    windows = (case["lo"] + case["hi"]) / 2 + (3500 if case["hot"] > 0 else 0)
    spread = case["sd"] / case["bin"] * 2 / (2 * case["eb"])  # of the predicted residual, in quantisation steps
    bits = max(1.02, 2.05 + math.log2(max(spread, 1e-3)))
    if case["hot"] > 0:
        bits += 1.0  # every hot pixel leaves four large residuals
    return windows * (289 * (3.0 if case["roi_coder"] else 4.0) + 6) + bins * bits / 8 + 1700


def work(case):
    px = case["P"] * case["H"] * case["W"]
    stream = _stream_bytes(case)
    sides = 2 if case["op"] == "roundtrip" else 1
    # binning, quantisation, prediction and the peak screen: about ten operations a pixel
    return {"bytes": case["n"] * sides * (4 * px + stream), "flops": 10.0 * case["n"] * sides * px}


def exact(case, seed):
    """Streams are bytes and have no such value.  The restored frames have: every bin's
    mean to the nearest multiple of 2 eb, spread over its pixels, with the pixels of the
    windows as they were."""
    if case["op"] not in ("decompress", "roundtrip"):
        return None
    frames, spots = _make(case, seed)
    _, _, spots = _wanted(case, spots, frames)
    (P, H, W), b, n = _geometry(case), case["bin"], case["n"]
    Hb, Wb = -(-H // b), -(-W // b)
    params = _params(case)
    restored = torch.empty((n, P, H, W), dtype=torch.float64, device="cuda")
    one = torch.nn.functional.pad(torch.ones((H, W), dtype=torch.float64, device="cuda"), (0, Wb * b - W, 0, Hb * b - H))
    inside = one.view(Hb, b, Wb, b).sum((1, 3))
    for k in range(n):
        x = torch.nn.functional.pad(frames[k].double(), (0, Wb * b - W, 0, Hb * b - H))
        q = torch.round(x.view(P, Hb, b, Wb, b).sum((2, 4)) / inside / (2.0 * case["eb"])) * (2.0 * case["eb"])
        restored[k] = q.repeat_interleave(b, 1).repeat_interleave(b, 2)[:, :H, :W]
    f, pn, r, c = spots
    flat, src = restored.view(-1), frames.view(-1)
    for dr in range(params.roi_h):
        for dc in range(params.roi_w):
            rr, cc = r + dr - params.roi_h // 2, c + dc - params.roi_w // 2
            ok = (rr >= 0) & (rr < H) & (cc >= 0) & (cc < W)
            at = ((f[ok] * P + pn[ok]) * H + rr[ok]) * W + cc[ok]
            flat[at] = src[at].double()
    if case["op"] == "decompress":
        return [restored, None]
    return [None, None, None, restored, None]
