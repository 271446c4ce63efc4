"""Workloads of the integral-histogram engine, as a user's program runs them.

Each case is one pass through the public entry points (``ihist.Plan``,
``ihist.Batch``, ``ihist_sequence_host``): the integral histogram of a frame
or of a batch of frames (Eq. 1), the region queries made on it (Eq. 2), the
window search, or the host-to-host pipeline of a frame sequence.  Plans,
batches and output buffers are kept between passes, as a program that
handles a video stream keeps them; every pass recomputes everything that it
returns.

``listed()``  the cases; ``draw(rng)``  one more case of the same ranges;
``prepare(case, seed)`` / ``run(state)``  inputs on the GPU, and one pass;
``work(case)``  bytes and operations that a pass cannot do without;
``exact(case, seed)``  the outputs from plain torch in 64-bit integers.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1711_01919_gb300 import ihist

LAYOUTS = {"bin": ihist.IHIST_BIN_MAJOR, "pixel": ihist.IHIST_PIXEL_MAJOR, "quad": ihist.IHIST_QUAD_MAJOR}
# the mix of a batch of uneven frames: (w, h) and bin counts
MIX_SIZES = ((320, 240), (640, 480), (1280, 720), (1920, 1080))
MIX_BINS = (16, 32, 64)
RING = 2  # histograms that a host sequence keeps on the device


def listed():
    return [
        # One small camera frame at a time, then the histograms of the
        # tracker's candidate regions: launches and latency count.
        {"name": "vga frame + queries", "kind": "frame", "h": 480, "w": 640, "bins": 32, "layout": "bin",
         "pixels": "uniform", "rects": 1000},
        # The same for one full-HD frame with fine bins, the common video size.
        {"name": "hd frame + queries", "kind": "frame", "h": 1080, "w": 1920, "bins": 64, "layout": "bin",
         "pixels": "gradient", "rects": 1000},
        # A region of interest cut from a larger frame: odd width and height,
        # a bin count that is no multiple of 4, rows that start unaligned.
        {"name": "ragged crop + queries", "kind": "frame", "h": 601, "w": 1021, "bins": 37, "layout": "bin",
         "pixels": "gradient", "rects": 300, "pad": 6},
        # Every pixel's histogram kept together, for many queries per frame.
        {"name": "hd pixel-major + queries", "kind": "frame", "h": 1080, "w": 1920, "bins": 64, "layout": "pixel",
         "pixels": "gradient", "rects": 10000},
        # A 4K frame in the layout that favours queries over the scan, with
        # bins by edges (dark tones binned finely, bright ones coarsely).
        {"name": "4k quad-major by edges", "kind": "frame", "h": 2160, "w": 3840, "bins": 64, "layout": "quad",
         "pixels": "gradient", "rects": 10000, "edges": True},
        # Joint colour histograms of an RGB frame, 4 x 4 x 4 bins.
        {"name": "hd joint rgb", "kind": "frame", "h": 1080, "w": 1920, "bins": 64, "layout": "bin",
         "pixels": "gradient", "rects": 0, "joint": True},
        # Live video from host memory: uploads double-buffered against the
        # scans, each frame's region histograms back on the host.
        {"name": "hd host sequence", "kind": "sequence", "frames": 16, "h": 1080, "w": 1920, "bins": 64,
         "layout": "bin", "pixels": "gradient", "rects": 1000},
        # Many cameras of uneven sizes and bin counts, served in one launch.
        {"name": "uneven batch", "kind": "batch", "frames": 256, "mix": 3, "layout": "bin", "pixels": "uniform",
         "rects": 0},
        # A stretch of full-HD video at once, with every frame's regions.
        {"name": "hd batch + queries", "kind": "batch", "frames": 64, "h": 1080, "w": 1920, "bins": 64,
         "layout": "bin", "pixels": "gradient", "rects": 1000},
        # The largest single frame: 64 megapixels, 32 GiB of counts.
        {"name": "64mp frame", "kind": "frame", "h": 8192, "w": 8192, "bins": 128, "layout": "bin",
         "pixels": "sinusoid", "rects": 0},
        # Dense region queries on a large resident histogram.
        {"name": "64mp dense queries", "kind": "queries", "h": 8192, "w": 8192, "bins": 128, "pixels": "sinusoid",
         "rects": 1 << 20},
        # Detection: every 64 x 64 window on a 4-pixel grid against a target.
        {"name": "hd window search", "kind": "window", "h": 1080, "w": 1920, "bins": 64, "layout": "bin",
         "pixels": "gradient", "win": 64, "stride": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["frame"] * 5 + ["batch"] * 2 + ["queries", "window", "sequence"])
    pixels = rng.choice(["uniform", "gradient", "sinusoid"])
    if kind == "batch":
        n = _log_int(rng, 2, 96)
        rects = rng.choice([0, _log_int(rng, 50, 2000)])
        if rng.random() < 0.5:
            return {"kind": kind, "frames": n, "mix": rng.randrange(1, 1 << 20),
                    "layout": rng.choice(["bin", "bin", "quad", "pixel"]), "pixels": pixels, "rects": rects}
        w = _log_int(rng, 160, 2600)
        w = rng.choice([w, (w + 15) // 16 * 16])
        layout = rng.choice(["bin", "bin", "quad", "pixel"])
        h, bins = _log_int(rng, 120, 1440), _log_int(rng, 8, 96)
        bins = (bins + 3) // 4 * 4 if layout == "quad" else bins
        return {"kind": kind, "frames": max(1, min(n, (3 << 30) // (h * w * bins))), "h": h, "w": w, "bins": bins,
                "layout": layout, "pixels": pixels, "rects": rects}
    h, w = _log_int(rng, 96, 4400), _log_int(rng, 96, 6000)
    w = rng.choice([w, (w + 15) // 16 * 16, (w + 3) // 4 * 4])
    bins = _log_int(rng, 8, 160)
    if kind == "queries":
        h, w = max(h, 512), max(w, 512)
        return {"kind": kind, "h": h, "w": w, "bins": bins, "pixels": pixels, "rects": _log_int(rng, 20000, 1 << 20)}
    if kind == "window":
        h, w = min(h, 2200), min(w, 3900)
        return {"kind": kind, "h": h, "w": w, "bins": min(bins, 96), "layout": rng.choice(["bin", "pixel"]),
                "pixels": pixels, "win": _log_int(rng, 16, min(96, h, w)), "stride": rng.choice([1, 2, 3, 4, 5, 8])}
    if kind == "sequence":
        h, w = min(h, 1100), min(w, 2000)
        return {"kind": kind, "frames": rng.randrange(4, 24), "h": h, "w": w, "bins": min(bins, 64),
                "layout": "bin", "pixels": pixels, "rects": _log_int(rng, 100, 2000)}
    layout = rng.choice(["bin", "bin", "pixel", "quad"])
    case = {"kind": kind, "h": h, "w": w, "bins": (bins + 3) // 4 * 4 if layout == "quad" else bins,
            "layout": layout, "pixels": pixels, "rects": rng.choice([0, _log_int(rng, 50, 20000)])}
    option = rng.choice(["", "", "pad", "edges", "joint"])
    if option == "pad":
        case["pad"] = rng.randrange(1, 64)
    elif option == "edges":
        case["edges"] = True
    elif option == "joint":
        case["joint"], case["bins"] = True, rng.choice([24, 64, 100])
    return case


# ------------------------------------------------------------------ inputs

def _frame(h, w, kind, gen, channels=0):
    """uint8 pixels on the GPU: i.i.d. bytes, a smooth ramp with noise of
    sigma 20, or slow waves with a little noise."""
    if channels:
        return torch.stack([_frame(h, w, kind, gen) for _ in range(channels)], dim=2).contiguous()
    if kind == "uniform":
        return torch.randint(0, 256, (h, w), dtype=torch.uint8, device="cuda", generator=gen)
    x = torch.arange(w, device="cuda", dtype=torch.float32)
    y = torch.arange(h, device="cuda", dtype=torch.float32)[:, None]
    if kind == "gradient":
        v = 127.5 * (x / max(w - 1, 1) + y / max(h - 1, 1))
        v = v + 20.0 * torch.randn((h, w), device="cuda", generator=gen)
    else:
        v = 128.0 + 50.0 * torch.sin(2 * math.pi * x / 997.0) + 40.0 * torch.sin(2 * math.pi * y / 1231.0)
        v = v + 25.0 * torch.sin(2 * math.pi * (x + y) / 313.0)
        v = v + (24.0 * torch.rand((h, w), device="cuda", generator=gen) - 12.0)
    return v.round_().clamp_(0, 255).to(torch.uint8)


def _rects(n, h, w, gen):
    """n inclusive rectangles x0, y0, x1, y1 with uniformly drawn corners."""
    x = torch.randint(0, w, (n, 2), device="cuda", generator=gen).sort(dim=1).values
    y = torch.randint(0, h, (n, 2), device="cuda", generator=gen).sort(dim=1).values
    return torch.stack([x[:, 0], y[:, 0], x[:, 1], y[:, 1]], dim=1).to(torch.int32).contiguous()


def _edges(bins):
    """bins + 1 increasing edges in [0, 256], finer at the dark end (1-wide
    bins where there are more than fit)."""
    n = min(bins, 250)
    e = [int(250.0 * (0.6 * k / n + 0.4 * (k / n) ** 2)) for k in range(n + 1)]
    for k in range(1, n + 1):
        e[k] = max(e[k], e[k - 1] + 1)
    return e


def _joint_bins(bins):
    return {24: [2, 4, 3], 64: [4, 4, 4], 100: [5, 5, 4]}[bins]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _one_input(case, gen):
    """The frame of a case (a view of wider rows when the case pads them)."""
    pad = case.get("pad", 0)
    f = _frame(case["h"], case["w"] + pad, case["pixels"], gen, 3 if case.get("joint") else 0)
    return f[:, pad // 2:pad // 2 + case["w"]] if pad else f


def _batch_shapes(case):
    """(h, w, bins) of every frame of a batch."""
    if "mix" not in case:
        return [(case["h"], case["w"], case["bins"])] * case["frames"]
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["frames"]):
        w, h = r.choice(MIX_SIZES)
        out.append((h, w, r.choice(MIX_BINS)))
    return out


def _batch_inputs(case, gen):
    shapes = _batch_shapes(case)
    frames = [_frame(h, w, case["pixels"], gen) for h, w, _ in shapes]
    rects = None
    if case["rects"]:
        rects = torch.stack([_rects(case["rects"], h, w, gen) for h, w, _ in shapes])
    return shapes, frames, rects


def _offsets(shapes):
    """Where each frame's counts start in one buffer (256-byte steps), and its length."""
    off, at = [], 0
    for h, w, b in shapes:
        off.append(at)
        at += (h * w * b + 63) // 64 * 64
    return off, at


def _sequence_inputs(case, gen):
    h, w = case["h"], case["w"]
    frames = torch.stack([_frame(h, w, case["pixels"], gen) for _ in range(case["frames"])]).cpu().pin_memory()
    return frames, _rects(case["rects"], h, w, gen)


def _target(plan_bins, area, gen):
    """A histogram of `area` pixels, as one taken from a patch."""
    t = torch.rand(plan_bins, device="cuda", generator=gen)
    return (t / t.sum() * area).to(torch.int32)


def _plan(case):
    layout = LAYOUTS[case.get("layout", "bin")]
    if case.get("edges"):
        return ihist.Plan(case["h"], case["w"], layout=layout, edges=_edges(case["bins"]))
    if case.get("joint"):
        return ihist.Plan(case["h"], case["w"], layout=layout, bins_per_channel=_joint_bins(case["bins"]))
    return ihist.Plan(case["h"], case["w"], case["bins"], layout)


# ------------------------------------------------------------ prepare / run

def prepare(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "batch":
        shapes, frames, rects = _batch_inputs(case, gen)
        off, total = _offsets(shapes)
        buf = torch.zeros(total, dtype=torch.int32, device="cuda")
        layout = LAYOUTS[case["layout"]]
        outs = [buf[o:o + h * w * b].view(ihist.out_shape(h, w, b, layout)) for o, (h, w, b) in zip(off, shapes)]
        batch = ihist.Batch(frames, [b for _, _, b in shapes], [layout] * len(shapes), outs=outs)
        rows = (torch.empty(case["rects"] * sum(b for _, _, b in shapes), dtype=torch.int32, device="cuda")
                if rects is not None else None)
        return {"kind": kind, "batch": batch, "buf": buf, "rects": rects, "rows": rows}
    plan = _plan(case)
    if kind == "sequence":
        frames, rects = _sequence_inputs(case, gen)
        h, w, n, nrects = case["h"], case["w"], case["frames"], case["rects"]
        return {"kind": kind, "plan": plan, "frames": frames, "rects": rects,
                "slots": torch.empty((2, h, w), dtype=torch.uint8, device="cuda"),
                "outs": torch.empty((RING, *plan.out_shape), dtype=torch.int32, device="cuda"),
                "rows": torch.empty((nrects, plan.nbins), dtype=torch.int32, device="cuda"),
                "host_rows": torch.empty((n, nrects, plan.nbins), dtype=torch.int32).pin_memory(),
                "copy": torch.cuda.Stream()}
    frame = _one_input(case, gen)
    s = {"kind": kind, "plan": plan, "frame": frame, "hist": plan.empty_output()}
    if kind == "window":
        s["target"] = _target(plan.nbins, case["win"] ** 2, gen)
        s["win"], s["stride"] = case["win"], case["stride"]
        ny, nx = ihist.window_grid(case["h"], case["w"], case["win"], case["win"], case["stride"])
        s["scores"] = torch.empty((ny, nx), dtype=torch.int32, device="cuda")
    elif case["rects"]:
        s["rects"] = _rects(case["rects"], case["h"], case["w"], gen)
        s["rows"] = torch.empty((case["rects"], plan.nbins), dtype=torch.int32, device="cuda")
    if kind == "queries":
        s["work"] = torch.empty(plan.query_work_bytes(case["rects"]), dtype=torch.uint8, device="cuda")
    if kind in ("queries", "window"):
        plan.compute(frame, s["hist"])  # the resident histogram that the pass reads
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        s["batch"].compute()
        if s["rects"] is None:
            return {"hist": s["buf"]}
        return {"hist": s["buf"], "rows": s["batch"].query_all(s["rects"], out=s["rows"])}
    plan = s["plan"]
    if kind == "frame":
        hist = plan.compute(s["frame"], s["hist"])
        if "rects" not in s:
            return {"hist": hist}
        return {"hist": hist, "rows": plan.query(hist, s["rects"], out=s["rows"])}
    if kind == "queries":
        return {"rows": plan.query_sorted(s["hist"], s["rects"], out=s["rows"], work=s["work"])}
    if kind == "window":
        return {"scores": plan.window_search(s["hist"], s["target"], s["win"], s["win"], s["stride"],
                                             out=s["scores"])}
    frames = s["frames"]
    ihist.ihist_sequence_host(plan.handle, frames.data_ptr(), frames.stride(0), frames.shape[0],
                              s["slots"].data_ptr(), s["outs"].data_ptr(), RING, s["rects"].data_ptr(),
                              s["rects"].shape[0], s["rows"].data_ptr(), s["host_rows"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream, s["copy"].cuda_stream)
    return {"hist": s["outs"], "host_rows": s["host_rows"]}


# ------------------------------------------------------------- work / exact

def _query_bytes(n, bins, words):
    """Rectangles in, rows out, and the four corner words of each (or all of H)."""
    return 16 * n + 4 * n * bins + min(16 * n * bins, 4 * words)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(case)
        words = sum(h * w * b for h, w, b in shapes)
        out = sum(h * w for h, w, _ in shapes) + 4 * words
        out += sum(_query_bytes(case["rects"], b, h * w * b) for h, w, b in shapes if case["rects"])
        return {"bytes": out, "flops": 2 * words}
    h, w, b = case["h"], case["w"], case["bins"]
    words = h * w * b
    if kind == "sequence":
        n = case["frames"]
        return {"bytes": n * (h * w + 4 * words + _query_bytes(case["rects"], b, words)), "flops": 2 * n * words}
    if kind == "queries":
        return {"bytes": _query_bytes(case["rects"], b, words), "flops": 3 * case["rects"] * b}
    if kind == "window":
        ny, nx = ihist.window_grid(h, w, case["win"], case["win"], case["stride"])
        return {"bytes": 4 * ny * nx + min(16 * ny * nx * b, 4 * words), "flops": 5 * ny * nx * b}
    out = h * w * (3 if case.get("joint") else 1) + 4 * words
    if case["rects"]:
        out += _query_bytes(case["rects"], b, words)
    return {"bytes": out, "flops": 2 * words}


def _bin_of(frame, case):
    """int64 bin of every pixel (-1: no bin)."""
    v = frame.to(torch.int64)
    if case.get("joint"):
        q = torch.zeros_like(v[..., 0])
        for c, n in enumerate(_joint_bins(case["bins"])):
            q = q * n + v[..., c] * n // 256
        return q
    if case.get("edges"):
        e = torch.tensor(_edges(case["bins"]), device=v.device)
        q = torch.bucketize(v, e, right=True) - 1
        return torch.where(q < len(e) - 1, q, torch.full_like(q, -1))
    return v * case["bins"] // 256


def _exact_hist(frame, case, bins):
    """H[b][y][x] in int64."""
    q = _bin_of(frame, case)
    out = torch.empty((bins, *q.shape), dtype=torch.int64, device=q.device)
    for b in range(bins):
        out[b] = (q == b).to(torch.int64).cumsum(0).cumsum(1)
    return out


def _laid_out(hist, layout):
    if layout == "pixel":
        return hist.permute(1, 2, 0).contiguous()
    if layout == "quad":
        b, h, w = hist.shape
        return hist.view(b // 4, 4, h, w).permute(0, 2, 3, 1).contiguous()
    return hist


def _exact_rows(hist, rects):
    """Eq. 2 on a bin-major int64 H: [n][bins]."""
    p = torch.nn.functional.pad(hist, (1, 0, 1, 0))
    x0, y0, x1, y1 = (rects[:, i].to(torch.int64) for i in range(4))
    return (p[:, y1 + 1, x1 + 1] - p[:, y0, x1 + 1] - p[:, y1 + 1, x0] + p[:, y0, x0]).t().contiguous()


def exact(case, seed):
    gen, kind = _gen(seed), case["kind"]
    if kind == "batch":
        shapes, frames, rects = _batch_inputs(case, gen)
        off, total = _offsets(shapes)
        if total > 1 << 31:
            return None
        buf = torch.zeros(total, dtype=torch.int64, device="cuda")
        rows = []
        for i, (h, w, b) in enumerate(shapes):
            hist = _exact_hist(frames[i], {"bins": b}, b)
            buf[off[i]:off[i] + h * w * b] = _laid_out(hist, case["layout"]).reshape(-1)
            if rects is not None:
                rows.append(_exact_rows(hist, rects[i]).reshape(-1))
        return {"hist": buf, "rows": torch.cat(rows)} if rects is not None else {"hist": buf}
    bins = case["bins"]
    if case["h"] * case["w"] * bins > 1 << 31:
        return None
    if kind == "sequence":
        frames, rects = _sequence_inputs(case, gen)
        ring, rows = [None] * RING, []
        for i in range(frames.shape[0]):
            hist = _exact_hist(frames[i].cuda(), case, bins)
            ring[i % RING] = _laid_out(hist, case["layout"])
            rows.append(_exact_rows(hist, rects))
        return {"hist": torch.stack(ring), "host_rows": torch.stack(rows)}
    hist = _exact_hist(_one_input(case, gen), case, bins)
    if kind == "window":
        target = _target(bins, case["win"] ** 2, gen).to(torch.int64)
        ny, nx = ihist.window_grid(case["h"], case["w"], case["win"], case["win"], case["stride"])
        p = torch.nn.functional.pad(hist, (1, 0, 1, 0))
        y = torch.arange(ny, device="cuda")[:, None] * case["stride"]
        x = torch.arange(nx, device="cuda")[None, :] * case["stride"]
        score = torch.zeros((ny, nx), dtype=torch.int64, device="cuda")
        for b in range(bins):
            c = (p[b][y + case["win"], x + case["win"]] - p[b][y, x + case["win"]]
                 - p[b][y + case["win"], x] + p[b][y, x])
            score += torch.minimum(c, target[b])
        return {"scores": score}
    out = {} if kind == "queries" else {"hist": _laid_out(hist, case["layout"])}
    if case.get("rects"):
        out["rows"] = _exact_rows(hist, _rects(case["rects"], case["h"], case["w"], gen))
    return out
