"""The work that is timed for this library: what a user's program has it do, by its public calls.

A case is a dict of plain values. `call` names what is called:

  run        ZnccContext.zncc_run on device images: cost, DT aggregation and WTA, fused
  host       ZnccContext.zncc_run_host: the same from page-locked host images to a host map
  batch      zncc_run_batch over pairs of uneven size
  steps      zncc_cost_volume, dt_aggregate and wta_disparity in turn on the caller's volume
  volume     zncc_cost_volume alone
  wta        wta_disparity of a stored volume
  stats      zncc_window_stats of one image

Sizes, disparity ranges, windows and DT parameters are those of the benchmark configurations
(320x96, 640x192, 1242x375, 1280x384, 1920x1080; D 32 to 256; windows 7 to 11; sigma_s 20,
sigma_r 0.1, three iterations). Images are synthetic stereo pairs: blurred noise seen through a
disparity map of slanted planes, with a gain, an offset, noise and two occluded bands.
Contexts keep their automatic launch shapes.
"""

import math

import numpy as np
import torch

from paper_2212_00476_gb300 import zncc as Z

STORAGE = {"f32": Z.ZNCC_F32, "f16": Z.ZNCC_F16, "i8": Z.ZNCC_I8}
TORCH = {"f32": torch.float32, "f16": torch.float16}

# pairs of a batch, in turn: (W, H, D, window)
UNEVEN = [(640, 192, 64, 7), (1242, 375, 64, 9), (640, 192, 128, 11), (1280, 384, 64, 9),
          (640, 192, 192, 9), (1242, 375, 128, 7), (1280, 384, 128, 11), (640, 192, 64, 9)]


def _case(name, call, w, h, d, win, iters=3, storage="f32", sigma_s=20.0, sigma_r=0.1, pairs=1):
    return {"name": name, "call": call, "w": w, "h": h, "d": d, "win": win, "iters": iters,
            "storage": storage, "sigma_s": sigma_s, "sigma_r": sigma_r, "pairs": pairs}


def listed():
    return [
        # the smallest call: a thumbnail-sized pair matched without aggregation (latency)
        _case("match_320x96_d32", "run", 320, 96, 32, 9, iters=0),
        # the small requests of the serving mix
        _case("run_640x192_d64", "run", 640, 192, 64, 9),
        # the paper-sized pair, the headline workload
        _case("run_1280x384_d128", "run", 1280, 384, 128, 9),
        # the driving-dataset size (odd in both directions) with half storage
        _case("run_1242x375_d128_f16", "run", 1242, 375, 128, 9, storage="f16"),
        # the paper's 8-bit storage, taken for its quarter of the memory
        _case("run_1280x384_d128_i8", "run", 1280, 384, 128, 9, storage="i8"),
        # the largest pair of the configurations: full HD, the deepest disparity range
        _case("run_1920x1080_d256", "run", 1920, 1080, 256, 11),
        # a camera loop: images from page-locked host memory, the map back to it
        _case("host_1280x384_d128", "host", 1280, 384, 128, 9),
        # pairs of uneven size processed together
        _case("batch_8_uneven", "batch", 0, 0, 0, 0, pairs=8),
        # the method step by step on a volume that the caller keeps
        _case("steps_1242x375_d128", "steps", 1242, 375, 128, 9),
        # the matching cost alone, for callers with an aggregation of their own
        _case("volume_1280x384_d128_f16", "volume", 1280, 384, 128, 9, storage="f16"),
        # the disparity map of a stored volume
        _case("wta_1280x384_d128", "wta", 1280, 384, 128, 9),
        # window sums and deviations of a full HD image
        _case("stats_1920x1080", "stats", 1920, 1080, 1, 11),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["run", "run", "run", "host", "batch", "steps", "volume", "wta", "stats"])
    if call == "batch":
        return {k: v for k, v in _case("", call, 0, 0, 0, 0, iters=rng.randint(1, 3), pairs=rng.randint(2, 8),
                                       sigma_s=rng.uniform(8.0, 40.0),
                                       storage=rng.choice(["f32", "f32", "f16"])).items() if k != "name"}
    w, h, d = _spread(rng, 160, 1920), _spread(rng, 64, 1080), _spread(rng, 16, 256)
    if rng.random() < 0.5:                                  # half of the widths as cameras have them
        w = max(16, w // 16 * 16)
    storage = rng.choice(["f32", "f32", "f16", "i8"] if call in ("run", "host") else ["f32", "f16"])
    if call in ("steps", "stats"):
        storage = "f32"
    iters = rng.choice([0, 1, 2, 3, 3]) if call in ("run", "host") else rng.randint(1, 3)
    c = _case("", call, w, h, d, rng.choice([3, 5, 7, 9, 9, 11, 13, 15]), iters=iters, storage=storage,
              sigma_s=rng.uniform(8.0, 40.0), sigma_r=rng.uniform(0.06, 0.25))
    return {k: v for k, v in c.items() if k != "name"}


# ---- inputs --------------------------------------------------------------------------------

def _blurred(g, h, w):
    """Uniform noise under a Gaussian blur of 1.5 pixels, scaled to 0..255."""
    v = torch.rand((h + 12, w + 12), generator=g, device="cuda")
    k = [math.exp(-0.5 * (i / 1.5) ** 2) for i in range(-6, 7)]
    v = sum(k[i] * v[i:i + h, :] for i in range(13))
    v = sum(k[i] * v[:, i:i + w] for i in range(13))
    return (v - v.min()) * (255.0 / (v.max() - v.min()).clamp_min(1e-9))


def _pair(w, h, d, seed):
    """A stereo pair (uint8 [h][w], device): left, and right seen through slanted planes."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    left = _blurred(g, h, w).round()
    n = 5
    p = torch.rand((n, 5), generator=g, device="cuda")
    xx = torch.arange(w, device="cuda", dtype=torch.float32)[None, :].expand(h, w)
    yy = torch.arange(h, device="cuda", dtype=torch.float32)[:, None].expand(h, w)
    sx, sy = p[:, 0] * w, p[:, 1] * h
    dist = torch.stack([(xx - sx[k]) ** 2 + (yy - sy[k]) ** 2 for k in range(n)])
    planes = torch.stack([(p[k, 2] - 0.5) * 0.5 * d / w * (xx - sx[k]) + (p[k, 3] - 0.5) * 0.5 * d / h * (yy - sy[k])
                          + (0.15 + 0.7 * p[k, 4]) * d for k in range(n)])
    disp = planes.gather(0, dist.argmin(0)[None])[0].round().clamp(0, max(d - 1, 0)).long()
    at = (torch.arange(w, device="cuda")[None, :] + disp).clamp(max=w - 1)
    right = left.gather(1, at)
    band = torch.rand((2,), generator=g, device="cuda") * 0.95 * w
    col = torch.arange(w, device="cuda", dtype=torch.float32)
    hidden = ((col >= band[0]) & (col < band[0] + w / 40)) | ((col >= band[1]) & (col < band[1] + w / 40))
    right = torch.where(hidden[None, :], _blurred(g, h, w), right)
    right = 0.9 * right + 10.0 + 2.0 * torch.randn((h, w), generator=g, device="cuda")
    return left.to(torch.uint8), right.round().clamp(0, 255).to(torch.uint8)


def _specs(case):
    if case["call"] == "batch":
        return [UNEVEN[i % len(UNEVEN)] for i in range(case["pairs"])]
    return [(case["w"], case["h"], case["d"], case["win"])]


def prepare(case, seed):
    call, specs = case["call"], _specs(case)
    s = {"case": case, "storage": STORAGE[case["storage"]]}
    s["ctx"] = [Z.ZnccContext(*spec) for spec in specs]
    if call == "wta":                                       # a stored volume of aggregated costs
        w, h, d, _ = specs[0]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        v = torch.rand((h, w, d), generator=g, device="cuda").mul_(2.0).sub_(1.0)
        s["cost"] = v.to(TORCH[case["storage"]])
    else:
        pairs = [_pair(w, h, d, 1000 * seed + i) for i, (w, h, d, _) in enumerate(specs)]
        s["left"], s["right"] = [p[0] for p in pairs], [p[1] for p in pairs]
    maps = [(h, w) for w, h, _, _ in specs]
    if call == "host":
        s["stream"] = torch.cuda.Stream()
        s["ctx"][0].set_stream(s["stream"])
        s["pinned"] = [t.cpu().pin_memory() for t in (s["left"][0], s["right"][0])]
        s["pinned"].append(torch.zeros(maps[0], dtype=torch.int16).pin_memory())
        s["host"] = [s["pinned"][0].numpy(), s["pinned"][1].numpy(), s["pinned"][2].numpy().view(np.uint16)]
    else:
        s["disp"] = [torch.zeros(m, dtype=torch.int16, device="cuda") for m in maps]
    if call in ("steps", "volume"):
        w, h, d, _ = specs[0]
        s["cost"] = torch.zeros((h, w, d), dtype=TORCH[case["storage"]], device="cuda")
    if call == "stats":
        s["sums"] = [torch.zeros(maps[0], dtype=t, device="cuda") for t in (torch.int32, torch.int32, torch.float32)]
    torch.cuda.synchronize()                                # the host call's stream is its own
    return s


def run(s):
    case, call, ctx, st = s["case"], s["case"]["call"], s["ctx"][0], s["storage"]
    dt = (case["sigma_s"], case["sigma_r"], case["iters"])
    if call == "run":
        ctx.zncc_run(s["left"][0], s["right"][0], s["disp"][0], *dt, st)
        return s["disp"][0]
    if call == "host":
        ctx.zncc_run_host(*s["host"], *dt, st)
        return s["pinned"][2]
    if call == "batch":
        Z.zncc_run_batch(s["ctx"], s["left"], s["right"], s["disp"], *dt, st)
        return s["disp"]
    if call == "wta":
        ctx.wta_disparity(s["cost"], s["disp"][0], st)
        return s["disp"][0]
    if call == "stats":
        ctx.zncc_window_stats(s["left"][0], *s["sums"])
        return s["sums"]
    ctx.zncc_cost_volume(s["left"][0], s["right"][0], s["cost"], st)
    if call == "volume":
        return s["cost"]
    ctx.dt_aggregate(s["left"][0], s["cost"], *dt, st)
    ctx.wta_disparity(s["cost"], s["disp"][0], st)
    return s["cost"], s["disp"][0]


def work(case):
    """Bytes that go in and come out; operations of the method per (pixel, disparity): a product
    and four additions of a running window sum, four for the normalisation, two for each of the
    4 * iters recursive passes, one comparison."""
    call, elem = case["call"], {"f32": 4, "f16": 2, "i8": 1}[case["storage"]]
    moved = ops = 0.0
    for w, h, d, win in _specs(case):
        pix, vol = w * h, w * h * d
        if call in ("run", "host", "batch"):
            moved += pix * (1 + 1 + 2)
            ops += vol * (9 + 8 * case["iters"] + 1)
        elif call == "steps":
            moved += pix * (1 + 1 + 2) + vol * elem
            ops += vol * (9 + 8 * case["iters"] + 1)
        elif call == "volume":
            moved += pix * 2 + vol * elem
            ops += vol * 9
        elif call == "wta":
            moved += vol * elem + pix * 2
            ops += vol
        else:
            moved += pix * (1 + 4 + 4 + 4)
            ops += pix * 15
    return {"bytes": moved, "flops": ops}


# ---- the same in 64 bits, by plain torch ---------------------------------------------------

def _padded(img, r, left):
    """The image with its edge pixels repeated r times on each side, and `left` more on the left."""
    h, w = img.shape
    ys = torch.arange(-r, h + r, device=img.device).clamp(0, h - 1)
    xs = torch.arange(-r - left, w + r, device=img.device).clamp(0, w - 1)
    return img[ys][:, xs].double()


def _box(v, l):
    """Sums over l x l windows (whole numbers far below 2^53: exact)."""
    c = torch.nn.functional.pad(v, (1, 0, 1, 0)).cumsum(0).cumsum(1)
    return c[l:, l:] - c[:-l, l:] - c[l:, :-l] + c[:-l, :-l]


def _cost(left, right, d, win):
    h, w = left.shape
    r, n = win // 2, float(win * win)
    lp, rp = _padded(left, r, 0), _padded(right, r, d - 1)
    sl, sr = _box(lp, win), _box(rp, win)
    vl, vr = n * _box(lp * lp, win) - sl * sl, n * _box(rp * rp, win) - sr * sr
    out = torch.empty((h, w, d), dtype=torch.float64, device=left.device)
    for k in range(d):
        at = d - 1 - k                                      # column of the centre x - k, x = 0
        p = _box(lp * rp[:, at:at + w + 2 * r], win)
        var = vl * vr[:, at:at + w]
        c = (n * p - sl * sr[:, at:at + w]) / var.clamp_min(1.0).sqrt()
        out[:, :, k] = torch.where(var > 0, c, torch.zeros_like(c))
    return out


def _aggregate(cost, guide, sigma_s, sigma_r, iters):
    k = math.exp(-1.0 / sigma_s)
    g = guide.double()
    v = cost
    for _ in range(iters):
        for axis in (1, 0):                                 # rows, then columns
            w = k * torch.exp(-(g.diff(dim=axis)).abs() / (255.0 * sigma_r))
            lines, w = v.movedim(axis, 0), w.movedim(axis, 0)[:, :, None]
            n = lines.shape[0]
            f = (1.0 - k) * lines
            for i in range(1, n):
                f[i].addcmul_(w[i - 1], f[i - 1])
            b = (1.0 - k) * f
            for i in range(n - 2, -1, -1):
                b[i].addcmul_(w[i], b[i + 1])
            v = b.movedim(0, axis)
    return v


def exact(case, seed):
    call = case["call"]
    if call not in ("steps", "volume", "stats"):
        return None                                         # maps of whole numbers
    w, h, d, win = _specs(case)[0]
    if w * h * d > 1.5e8:                                   # several 64-bit volumes: too long
        return None
    left, right = _pair(w, h, d, 1000 * seed)
    if call == "stats":
        r, n = win // 2, float(win * win)
        p = _padded(left, r, 0)
        s, q = _box(p, win), _box(p * p, win)
        var = n * q - s * s
        inv = torch.where(var > 0, var.clamp_min(1.0).rsqrt(), torch.zeros_like(var))
        return [None, None, inv]
    c = _cost(left, right, d, win)
    if call == "volume":
        return c
    return _aggregate(c, left, case["sigma_s"], case["sigma_r"], case["iters"]), None
