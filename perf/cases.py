"""Performance cases of the census template matcher, through the Python binding a user calls.

Each case is one call (or one request burst) of the library as a program in service makes it:
single frames on a stream, captured batches, batches whose images start in host memory, the
serving loop, the plain census and the auto-rectification search.  Inputs are synthetic stereo
pairs rendered on the GPU from the seed: blurred noise (sigma 1.5) as background, every box with
a texture of its own at a planted disparity, gain, offset and noise on the right image -- the
recipe of the library's own workloads.  Every state has its own images and boxes, so repeated
passes over several states run on data that left the cache.

A case is a dict of plain values:
  entry   "frame" (match_boxes, then box_points when "points"), "batch" (match_batch, captured
          graph), "host" (match_batch_host_packed, copying or mapped), "serve" (Server),
          "census" (census_build), "rect" (auto_rect)
  W, H    image size;  frames: frames per call;  boxes: boxes per frame (mean with "poisson")
  side_lo, side_hi: log-uniform box sides;  params, and what each entry names below.
"""
import math

import numpy as np
import torch

from paper_2604_07980_gb300 import binding as B

F_PX, BASELINE_M = 2000.0, 0.30   # truck camera: focal length (px), stereo baseline (m)

# Matching parameters by name: the library's workload configurations, and "rows", a camera pair
# whose rectification leaves a row of vertical error (vertical search, small window).
PARAMS = {
    "pair": dict(win_w=7, win_h=7, far_side_px=0, close_factor=1, far_dmin=0, far_dmax=63, close_dmin=0,
                 close_dmax=63, dy_min=0, dy_max=0, grid_g=3, agg_nmin=3, agg_mode=0),
    "frame": dict(win_w=9, win_h=7, far_side_px=40, close_factor=2, far_dmin=0, far_dmax=31, close_dmin=0,
                  close_dmax=127, dy_min=0, dy_max=0, grid_g=4, agg_nmin=6, agg_mode=0),
    "wide": dict(win_w=9, win_h=7, far_side_px=40, close_factor=2, far_dmin=0, far_dmax=127, close_dmin=0,
                 close_dmax=63, dy_min=0, dy_max=0, grid_g=4, agg_nmin=6, agg_mode=0),
    "large": dict(win_w=9, win_h=7, far_side_px=40, close_factor=2, far_dmin=0, far_dmax=63, close_dmin=0,
                  close_dmax=127, dy_min=0, dy_max=0, grid_g=5, agg_nmin=9, agg_mode=1),
    "rows": dict(win_w=5, win_h=5, far_side_px=40, close_factor=2, far_dmin=-2, far_dmax=29, close_dmin=0,
                 close_dmax=79, dy_min=-1, dy_max=1, grid_g=3, agg_nmin=3, agg_mode=0),
}
COMMON = dict(sentinel=1, pts_side=16, min_pts=16, fb_tol=1, agg_tau_d=1.0, trim_frac=0.2, max_occluders=16)


def _params(case):
    return {**COMMON, **PARAMS[case["params"]]}


def listed():
    return [
        # the smallest call: one VGA pair, four detections, latency of the launches
        dict(name="pair640", entry="frame", W=640, H=480, frames=1, boxes=4, poisson=False, side_lo=48, side_hi=48,
             strips=False, params="pair", points=False),
        # one camera frame of the usual size, detections to 3-D points (a driving stack, frame by frame)
        dict(name="frame1080_points", entry="frame", W=1920, H=1080, frames=1, boxes=64, poisson=False, side_lo=12,
             side_hi=400, strips=False, params="frame", points=True),
        # odd frame size, vertical search, the small census window: an imperfectly rectified pair
        dict(name="frame719_rows", entry="frame", W=1279, H=719, frames=1, boxes=48, poisson=False, side_lo=12,
             side_hi=300, strips=False, params="rows", points=False),
        # a small captured batch: four 720p cameras at one instant
        dict(name="lane4x720", entry="batch", W=1280, H=720, frames=4, boxes=60, poisson=True, side_lo=12, side_hi=400,
             strips=False, params="frame"),
        # the batched workload: 32 frames, partly occluded boxes
        dict(name="batch32x1200", entry="batch", W=1920, H=1200, frames=32, boxes=40, poisson=True, side_lo=12,
             side_hi=600, strips=True, params="wide"),
        # the largest: 4K frames with many boxes, trimmed mean over 25 blocks
        dict(name="batch8x2160", entry="batch", W=3840, H=2160, frames=8, boxes=256, poisson=False, side_lo=12,
             side_hi=800, strips=False, params="large"),
        # the batched workload from page-locked host images, the device reading what it needs
        dict(name="mapped32x1200", entry="host", W=1920, H=1200, frames=32, boxes=40, poisson=True, side_lo=12,
             side_hi=600, strips=True, params="wide", mapped=True),
        # host images copied whole (hosts that want their buffers back at once)
        dict(name="copied8x1200", entry="host", W=1920, H=1200, frames=8, boxes=40, poisson=True, side_lo=12,
             side_hi=600, strips=True, params="wide", mapped=False),
        # a burst of sixteen 1080p frames through the serving loop, submit to last result
        dict(name="serve16x1080", entry="serve", W=1920, H=1080, frames=16, boxes=60, poisson=True, side_lo=12,
             side_hi=400, strips=False, params="frame"),
        # the census of a whole image, for callers with a search of their own
        dict(name="census1200", entry="census", W=1920, H=1200, frames=1, factor=1, win_w=9, win_h=7),
        # the same at half resolution on an odd 4K image with the square window
        dict(name="census2159_half", entry="census", W=3839, H=2159, frames=1, factor=2, win_w=7, win_h=7),
        # the vertical-offset search on a 128-row band of a 1920x1200 pair
        dict(name="rect128", entry="rect", W=1920, H=1200, frames=1, band=128, disparities=64, offsets=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges: sizes log-uniform from 320 to 3840 columns (odd ones among
    them), 1 to 32 frames within the largest listed case's pixels and boxes."""
    entry = rng.choice(["frame", "frame", "batch", "batch", "host", "serve", "census", "rect"])
    W = int(_log(rng, 320, 3840))
    H = max(200, min(2160, int(W * rng.uniform(0.5, 0.75))))
    if entry in ("batch", "host", "serve") and rng.random() < 0.7:
        W, H = (W + 15) // 16 * 16, (H + 7) // 8 * 8  # most cameras' sizes
    if entry == "census":
        w = rng.choice([(9, 7), (7, 7), (5, 5), (11, 5)])
        return dict(entry=entry, W=W, H=H, frames=1, factor=rng.choice([1, 1, 2, 2, 3]), win_w=w[0], win_h=w[1])
    if entry == "rect":
        return dict(entry=entry, W=W, H=H, frames=1, band=int(_log(rng, 32, min(H, 256))),
                    disparities=rng.choice([32, 48, 64, 96]), offsets=rng.randint(1, 5))
    params = rng.choice(["frame", "wide", "large", "rows"])
    hi = int(min(W, H) * rng.uniform(0.3, 0.6))
    most = int(min(60e6 / (W * H), 32))
    frames = 1 if entry == "frame" else max(1, min(most, int(_log(rng, 1, 33))))
    boxes = max(1, min(int(_log(rng, 4, 257)), 1600 // frames))
    case = dict(entry=entry, W=W, H=H, frames=frames, boxes=boxes, poisson=frames > 1, side_lo=12, side_hi=max(hi, 24),
                strips=rng.random() < 0.4, params=params)
    if entry == "frame":
        case["points"] = rng.random() < 0.5
    if entry == "host":
        case["mapped"] = rng.random() < 0.6
    return case


# ----------------------------------------------------------------------------- inputs

def _texture(gen, h, w):
    """Blurred white noise of mean 128 and deviation 40, float32 on the GPU."""
    t = torch.arange(-5, 6, dtype=torch.float32, device="cuda")
    g = torch.exp(-t * t / (2 * 1.5 ** 2))
    g = g / g.sum()
    a = torch.randn((1, 1, h + 10, w + 10), generator=gen, device="cuda")
    a = torch.nn.functional.conv2d(a, g.view(1, 1, 1, 11))
    a = torch.nn.functional.conv2d(a, g.view(1, 1, 11, 1))[0, 0]
    return (a - a.mean()) / a.std() * 40 + 128


def _boxes(case, rng, fi):
    """Boxes [n, 5] and their true disparities of one frame: log-uniform sides, every fifth box with an
    occluding strip (its bottom edge lower, nearer) when "strips".  The frame's count (Poisson) belongs to
    the case, everything else to the seed."""
    W, H, p = case["W"], case["H"], _params(case)
    n = case["boxes"]
    if case["poisson"]:
        n = min(int(np.random.default_rng([n, case["frames"], fi]).poisson(n)), 2 * n + 10)
    boxes, d = [], []
    for _ in range(n):
        side = math.exp(rng.uniform(math.log(case["side_lo"]), math.log(case["side_hi"] + 1e-3)))
        a = rng.uniform(0.5, 1.5) if case["side_hi"] > case["side_lo"] else 1.0
        w, h = (side / a, side) if a >= 1 else (side, side * a)
        w, h = int(max(2, min(round(w), W))), int(max(2, min(round(h), H)))
        x0, y0 = int(rng.integers(0, W - w + 1)), int(rng.integers(0, H - h + 1))
        far = max(w, h) < p["far_side_px"]
        k = 1 if far else p["close_factor"]
        hi = (p["far_dmax"] if far else p["close_dmax"]) * k
        boxes.append([x0, y0, x0 + w, y0 + h, fi])
        d.append(rng.uniform(0.5, max(hi - 3, 1)))
    if case["strips"]:
        for i in range(0, n, 5):
            x0, y0, x1, y1, _ = boxes[i]
            w = x1 - x0
            sw = min(max(2, int(round(rng.uniform(0.1, 0.3) * w))), w)
            sx = int(rng.integers(x0, x1 - sw + 1))
            boxes.append([sx, y0, sx + sw, min(y1 + int(rng.integers(1, 11)), H), fi])
            d.append(d[i] + rng.uniform(5, 20))
    return boxes, d


def _pair(W, H, boxes, d, gen, rng, shift=0):
    """One rendered stereo pair (uint8 [2, H, W] on the GPU): boxes painted nearest last (ascending bottom
    edge), in the right image moved left by their disparity with bilinear sampling; `shift` rows lower on
    the left (a vertical misalignment)."""
    bg, own = _texture(gen, H + 16, W), _texture(gen, H + 16, W + 2)
    left, right = bg[8 - shift:8 - shift + H].clone(), bg[8:8 + H].clone()
    for i in sorted(range(len(boxes)), key=lambda j: (boxes[j][3], j)):
        x0, y0, x1, y1 = boxes[i][:4]
        w, h = x1 - x0, y1 - y0
        tx, ty = int(rng.integers(0, W - w + 1)), int(rng.integers(0, H - h + 1))
        tex = own[ty:ty + h, tx:tx + w + 2]
        left[y0:y1, x0:x1] = tex[:, :w]
        r0, r1 = max(math.ceil(x0 - d[i]), 0), math.ceil(x1 - d[i])
        if r1 > r0:
            u = r0 - x0 + d[i]
            iu = int(math.floor(u))
            n = min(r1 - r0, w + 1 - iu)
            f = u - iu
            right[y0:y1, r0:r0 + n] = tex[:, iu:iu + n] * (1 - f) + tex[:, iu + 1:iu + 1 + n] * f
    gain, offset = float(rng.uniform(0.8, 1.2)), float(rng.uniform(-20, 20))
    right = gain * right + offset + 2.0 * torch.randn(right.shape, generator=gen, device="cuda")
    return torch.stack([left, right]).round_().clamp_(0, 255).to(torch.uint8)


def _inputs(case, seed):
    """Images [frames, 2, H, W] (uint8, on the GPU) and boxes [n, 5] (int32, host) of a matching case."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.default_rng([int(seed), 5])
    images = torch.empty((case["frames"], 2, case["H"], case["W"]), dtype=torch.uint8, device="cuda")
    boxes = []
    for f in range(case["frames"]):
        b, d = _boxes(case, rng, f)
        images[f] = _pair(case["W"], case["H"], b, d, gen, rng)
        boxes += b
    return images, np.array(boxes, np.int32).reshape(-1, 5)


def _capacity(case):
    """Boxes a context is made for: the count itself, or what Poisson counts and strips stay below."""
    n = case["boxes"] * (1.3 if case["strips"] else 1.0)
    per = case["boxes"] if not case["poisson"] and not case["strips"] else 2 * (2 * case["boxes"] + 10)
    return int(min(case["frames"] * per, case["frames"] * n + 10 * math.sqrt(case["frames"] * n) + 40))


def _calibration(W, H):
    """Reprojection of a centred principal point and a camera mounted 1.6 m up, 1.2 m ahead of the axle."""
    Q = [[1, 0, 0, -(W - 1) / 2], [0, 1, 0, -(H - 1) / 2], [0, 0, 0, F_PX], [0, 0, 1 / BASELINE_M, 0]]
    T = [[0, 0, 1, 1.2], [-1, 0, 0, 0.1], [0, -1, 0, 1.6]]
    return dict(Q=Q, T=T, disp_var=0.04, f_px=F_PX, baseline_m=BASELINE_M, width=W, height=H)


class _State:
    def __init__(self, case):
        self.case = case

    def close(self):
        for name in ("ctx", "server"):
            if getattr(self, name, None) is not None:
                torch.cuda.synchronize()
                getattr(self, name).close()

    __del__ = close


def _rect_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 29)
    rng = np.random.default_rng([int(seed), 6])
    # objects across the band at many depths, the right image a few rows off
    b, d = [], []
    for _ in range(60):
        w, h = int(rng.integers(40, max(41, case["W"] // 6))), int(rng.integers(30, max(31, case["H"] // 3)))
        x0, y0 = int(rng.integers(0, case["W"] - w + 1)), int(rng.integers(0, case["H"] - h + 1))
        b.append([x0, y0, x0 + w, y0 + h])
        d.append(float(rng.uniform(3, case["disparities"] - 2)))
    return _pair(case["W"], case["H"], b, d, gen, rng, shift=int(rng.integers(-2, 3)))


def prepare(case, seed):
    s = _State(case)
    W, H = case["W"], case["H"]
    if case["entry"] == "census":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) * 7919 + 31)
        s.image = _texture(gen, H, W).round_().clamp_(0, 255).to(torch.uint8)
        return s
    if case["entry"] == "rect":
        s.image = _rect_inputs(case, seed)
        y0 = (H - case["band"]) // 2
        s.roi = (0, y0, W, y0 + case["band"])
        return s
    images, boxes = _inputs(case, seed)
    s.boxes = boxes
    n, frames = _capacity(case), case["frames"]
    assert len(boxes) <= n, (len(boxes), n)
    if case["entry"] == "serve":
        s.images = images.cpu().pin_memory()
        s.server = B.Server(_params(case), max_width=W, max_height=H, max_boxes_per_frame=2 * (2 * case["boxes"] + 10))
        s.frame_boxes = [boxes[boxes[:, 4] == f] for f in range(frames)]
    elif case["entry"] == "host":
        s.images = images.cpu().pin_memory()
        s.ctx = B.Context(_params(case), frames, W, H, n)
    else:
        s.images = images
        s.ctx = B.Context(_params(case), frames, W, H, n)
        if case["entry"] == "frame":
            s.boxes_dev = torch.from_numpy(boxes).cuda()
            s.geo, s.n_geo = B.geometries_to_device([_calibration(W, H)])
        else:
            s.batch = B.DeviceBatch([(im[0], im[1]) for im in images], boxes, [(F_PX, BASELINE_M)] * frames)
    return s


def run(s):
    case = s.case
    if case["entry"] == "census":
        return B.census_build(s.image, case["factor"], case["win_w"], case["win_h"])
    if case["entry"] == "rect":
        delta, counts = B.auto_rect(s.image[0], s.image[1], s.roi, 0, case["disparities"] - 1, -case["offsets"],
                                    case["offsets"], 2)
        return {"delta": delta, "counts": counts}
    if case["entry"] == "frame":
        out = s.ctx.match_boxes(s.images[0, 0], s.images[0, 1], s.boxes_dev, F_PX, BASELINE_M)
        if case["points"]:
            out["points"] = B.box_points(s.boxes_dev, out["disp"], out["flags"], s.geo, s.n_geo)
        return out
    if case["entry"] == "batch":
        return s.ctx.match_batch(s.batch, use_graph=True)
    if case["entry"] == "host":
        return s.ctx.match_batch_host_packed(s.images.numpy(), s.boxes, F_PX, BASELINE_M, mapped=case["mapped"])
    tags = []
    for f in range(case["frames"]):
        tags.append(s.server.submit(s.images[f, 0], s.images[f, 1], s.frame_boxes[f], F_PX, BASELINE_M))
    done = {r["tag"]: r for r in s.server.wait_all()}
    done = [done[t] for t in tags]
    assert all(r["status"] == 0 for r in done)
    return {key: np.concatenate([r[key] for r in done]) for key in ("disp", "depth", "flags")}


# ----------------------------------------------------------------------------- least work

def work(case):
    """Bytes: image bytes read once and results written once; matching needs only the rows and columns
    its blocks sample and search (their expectation over the box sizes).  Operations: two 32-bit xors, two
    population counts and one add per 64-bit cost evaluation, one compare per census comparison."""
    W, H = case["W"], case["H"]
    if case["entry"] == "census":
        k = case["factor"]
        codes = -(-W // k) * -(-H // k)
        return {"bytes": codes * (1 + 8), "flops": codes * (case["win_w"] * case["win_h"] - 1)}
    if case["entry"] == "rect":
        rows, nd, deltas = case["band"], case["disparities"], 2 * case["offsets"] + 1
        codes = W * (2 * rows + 2 * case["offsets"])
        return {"bytes": codes + 8 * deltas, "flops": 5 * 2 * W * rows * nd * deltas + 62 * codes}
    p = _params(case)
    ndy = p["dy_max"] - p["dy_min"] + 1
    lo, hi = math.log(case["side_lo"]), math.log(case["side_hi"] + 1e-3)
    evals = codes = pixels = 0.0
    steps = 64
    for i in range(steps):  # expectation over the log-uniform side (mean aspect about 1)
        side = math.exp(lo + (hi - lo) * (i + 0.5) / steps)
        far = side < p["far_side_px"]
        k, g = (1, 1) if far else (p["close_factor"], p["grid_g"])
        nd = (p["far_dmax"] - p["far_dmin"] if far else p["close_dmax"] - p["close_dmin"]) + 1
        w, h = side / k, 0.85 * side / k
        nx, ny = min(w / g, p["pts_side"]), min(h / g, p["pts_side"])
        evals += 2 * g * g * nx * ny * nd * ndy / steps
        rows = min(h, g * ny)
        codes += 2 * rows * (w + nd) / steps
        pixels += 2 * min(h, rows * p["win_h"]) * (w + nd) / steps
    n = case["boxes"] * case["frames"] * (1.2 if case["strips"] else 1.0)
    pixels = min(n * pixels, 2 * W * H * case["frames"])
    if case["entry"] == "host" and not case["mapped"]:
        pixels = 2 * W * H * case["frames"]
    out = 20 + 9 + (32 if case.get("points") else 0)
    return {"bytes": pixels + n * out, "flops": 5 * n * evals + n * codes * (p["win_w"] * p["win_h"] - 1)}


# ----------------------------------------------------------------------------- 64-bit values

def _popcount_table():
    t = torch.zeros(65536, dtype=torch.int16, device="cuda")
    for b in range(16):
        t += ((torch.arange(65536, device="cuda") >> b) & 1).to(torch.int16)
    return t


def _census(img, k, win_w, win_h):
    """Census codes of I(k x, k y) as int64 (raster order, sentinel on top), 0 where the window leaves it."""
    g = img[::k, ::k].to(torch.int16)
    h, w = g.shape
    sx, sy = win_w // 2, win_h // 2
    out = torch.zeros((h, w), dtype=torch.int64, device=img.device)
    if h <= 2 * sy or w <= 2 * sx:
        return out
    c = g[sy:h - sy, sx:w - sx]
    code = torch.ones(c.shape, dtype=torch.int64, device=img.device)
    for j in range(win_h):
        for i in range(win_w):
            code = (code << 1) | (g[j:j + c.shape[0], i:i + c.shape[1]] > c).to(torch.int64)
    out[sy:h - sy, sx:w - sx] = code
    return out


def _blocks_of(p, W, H, boxes):
    """Points of every searchable block of one frame: (box, k, X, Y) with the usable points, and the
    boxes' kinds; occluded points (in a nearer overlapping box) left out."""
    r = np.stack([boxes[:, 0].clip(0), boxes[:, 1].clip(0), boxes[:, 2].clip(max=W), boxes[:, 3].clip(max=H)], 1)
    sx, sy = p["win_w"] // 2, p["win_h"] // 2
    got = []
    for i, (x0, y0, x1, y1) in enumerate(r.tolist()):
        if x1 <= x0 or y1 <= y0:
            continue
        far = max(x1 - x0, y1 - y0) < p["far_side_px"]
        k, g = (1, 1) if far else (p["close_factor"], p["grid_g"])
        occ = [j for j in range(len(r)) if j != i and r[j, 3] > y1 and min(r[j, 2], x1) > max(r[j, 0], x0)
               and min(r[j, 3], y1) > max(r[j, 1], y0)]
        occ = r[sorted(occ, key=lambda j: (-r[j, 3], j))[:p["max_occluders"]]]
        a0, a1, b0, b1 = -(-x0 // k), -(-x1 // k), -(-y0 // k), -(-y1 // k)
        Wk, Hk = -(-W // k), -(-H // k)

        def cells(lo, hi, q):
            c0, c1 = lo + q * (hi - lo) // g, lo + (q + 1) * (hi - lo) // g
            n = min(c1 - c0, p["pts_side"])
            return c0 + ((2 * np.arange(n) + 1) * (c1 - c0)) // (2 * max(n, 1))

        for slot in range(g * g):
            X, Y = np.meshgrid(cells(a0, a1, slot % g), cells(b0, b1, slot // g))
            X, Y = X.ravel(), Y.ravel()
            ok = (X >= sx) & (X + sx < Wk) & (Y >= sy) & (Y + sy < Hk)
            if len(occ):
                ok &= ~((k * X >= occ[:, :1]) & (k * X < occ[:, 2:3]) & (k * Y >= occ[:, 1:2])
                        & (k * Y < occ[:, 3:4])).any(0)
            if ok.sum() >= p["min_pts"]:
                got.append((i, far, X[ok], Y[ok]))
    return got


def _search(CL, CR, X, Y, mask, dmin, dmax, dy_min, dy_max, table):
    """Forward costs' first minimum, its parabola vertex (64 bits) and the backward minimum, per block."""
    nd = dmax - dmin + 1
    cand = [(dy, d) for dy in range(dy_min, dy_max + 1) for d in range(dmin, dmax + 1)]
    D = torch.tensor([c[1] for c in cand], device="cuda")
    DY = torch.tensor([c[0] for c in cand], device="cuda")
    H, W = CL.shape

    def at(C, x, y):
        ok = (x >= 0) & (x < W) & (y >= 0) & (y < H)
        return torch.where(ok, C[y.clamp(0, H - 1), x.clamp(0, W - 1)], 0)

    def costs(q, C, x, y):
        v = q[:, :, None] ^ at(C, x, y)
        n = sum(table[(v >> s) & 0xffff] for s in (0, 16, 32, 48))
        return (n * mask[:, :, None].to(torch.int16)).sum(1, dtype=torch.int64)

    def first(c):
        return ((c * len(cand) + torch.arange(len(cand), device="cuda")).min(1).values) % len(cand)

    cf = costs(at(CL, X, Y), CR, X[:, :, None] - D, Y[:, :, None] + DY)
    b = first(cf)
    d, dy = D[b], DY[b]
    QX, QY = X - d[:, None], Y + dy[:, None]
    cb = costs(at(CR, QX, QY), CL, QX[:, :, None] + D, QY[:, :, None] - DY)
    db = D[first(cb)]
    row = torch.arange(len(b), device="cuda")
    inner = (d > dmin) & (d < dmax)
    s_m, s_0, s_p = (cf[row, (b + o).clamp(0, len(cand) - 1)].double() for o in (-1, 0, 1))
    den = 2 * (s_p + s_m - 2 * s_0)
    off = torch.where(inner & (den != 0), (s_p - s_m) / torch.where(den == 0, 1.0, den), 0.0)
    return (d.double() - off).cpu().numpy(), (db - d).abs().cpu().numpy()


def _aggregate(p, far, v):
    """The box's disparity from its consistent blocks' (None: none)."""
    if far:
        return v[0] if len(v) == 1 else None
    v = np.sort(np.array(v, np.float64))
    if not len(v):
        return None
    start = best = 0
    length = 1
    for i in range(1, len(v)):
        if not v[i] - v[i - 1] < p["agg_tau_d"]:
            start = i
        if i - start + 1 > length:
            length, best = i - start + 1, start
    if length < p["agg_nmin"]:
        return None
    run = v[best:best + length]
    if p["agg_mode"] == 0:
        return float(np.median(run))
    t = int(math.floor(p["trim_frac"] * length))
    return float(run[t:length - t].mean())


def exact(case, seed):
    """Disparities, depths and points of the matching cases by their definition, in 64 bits; flags, codes
    and counts are whole numbers and have no such value."""
    if case["entry"] in ("census", "rect"):
        return None
    p = _params(case)
    W, H = case["W"], case["H"]
    images, boxes = _inputs(case, seed)
    table = _popcount_table()
    disp = np.full(len(boxes), np.nan)
    for f in range(case["frames"]):
        mine = np.flatnonzero(boxes[:, 4] == f)
        blocks = _blocks_of(p, W, H, boxes[mine])
        found = {i: (b[1], []) for b in blocks for i in [b[0]]}
        for far in (True, False):
            some = [b for b in blocks if b[1] == far]
            if not some:
                continue
            k = 1 if far else p["close_factor"]
            CL, CR = (_census(images[f, q], k, p["win_w"], p["win_h"]) for q in (0, 1))
            lo, hi = (p["far_dmin"], p["far_dmax"]) if far else (p["close_dmin"], p["close_dmax"])
            for c in range(0, len(some), 128):
                part = some[c:c + 128]
                X, Y, mask = (np.zeros((len(part), p["pts_side"] ** 2), np.int64) for _ in range(3))
                for r, b in enumerate(part):
                    n = len(b[2])
                    X[r, :n], Y[r, :n], mask[r, :n] = b[2], b[3], 1
                X, Y, mask = (torch.from_numpy(a).cuda() for a in (X, Y, mask))
                d, off = _search(CL, CR, X, Y, mask, lo, hi, p["dy_min"], p["dy_max"], table)
                for b, v, o in zip(part, d, off):
                    if o <= p["fb_tol"]:
                        found[b[0]][1].append(v * k)
        for i, (far, v) in found.items():
            got = _aggregate(p, far, v)
            if got is not None and got > 0:
                disp[mine[i]] = got
    fb = float(np.float32(F_PX)) * float(np.float32(BASELINE_M))
    out = {"disp": disp, "depth": fb / disp, "flags": None}
    if case.get("points"):
        c = _calibration(W, H)
        Q, T = np.array(c["Q"], np.float32).astype(np.float64), np.array(c["T"], np.float32).astype(np.float64)
        u = (boxes[:, 0].clip(0) + boxes[:, 2].clip(max=W) - 1) / 2
        v = (boxes[:, 1].clip(0) + boxes[:, 3].clip(max=H) - 1) / 2
        X = Q @ np.stack([u, v, disp, np.ones(len(u))])
        cam = X[:3] / X[3]
        car = T @ np.concatenate([cam, np.ones((1, len(u)))])
        var = cam[2] ** 4 * float(np.float32(c["disp_var"])) / fb ** 2
        out["points"] = np.concatenate([cam, car, [var], X[3:4]]).T
    return out
