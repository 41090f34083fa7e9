"""Measured cases: the work a user of this library has it do, through its public entry points.

Each case names one call (or one pair of calls) a program makes in steady state: a forward on one
image, a batched forward, a training step, the gradient alone, a standalone integral histogram, the
merge of a bracketed exposure. `prepare` makes the inputs on the GPU and holds the context a program
keeps; `run` makes the calls; `exact` states the operator in 64 bits with plain torch.
"""
import functools
import math

import numpy as np
import torch

import paper_2102_01289_gb300 as tm

DTYPES = {"f32": torch.float32, "f16": torch.float16, "u8": torch.uint8}
EPS, SAT = float(np.float32(0.1)), float(np.float32(0.6))  # the paper's values as the library holds them


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # a thumbnail or preview: the smallest call, where launches and latency count
        dict(name="forward-512x384", kind="forward", width=512, height=384, bins=32, fields="4/16/64",
             src="f32", dst="f32"),
        # a photograph of odd size shown on a display: uint8 out, ragged rows
        dict(name="forward-1365x1023-u8", kind="forward", width=1365, height=1023, bins=64, fields="8/32/128",
             src="f32", dst="u8"),
        # one frame of a half-precision video
        dict(name="forward-1080p-f16", kind="forward", width=1920, height=1080, bins=32, fields="8/32/128",
             src="f16", dst="f16"),
        # the headline: one 12 MP photograph, 64 bins, three fields
        dict(name="forward-12mp", kind="forward", width=4000, height=3000, bins=64, fields="8/32/128",
             src="f32", dst="f32"),
        # the paper's own setting at 12 MP: five fields halving from the whole image, five bins
        dict(name="forward-12mp-pyramid", kind="forward", width=4000, height=3000, bins=5, fields="pyramid5",
             src="f32", dst="f32"),
        # a clip processed at once: 120 half-precision 1080p frames
        dict(name="batch-video-120", kind="batch", images=120, width=1920, height=1080, uneven=0, bins=32,
             fields="8/32/128", src="f16", dst="f16"),
        # a folder of photographs of all sizes from 640 x 480 to 4096 x 3072
        dict(name="batch-uneven-16", kind="batch", images=16, width=4096, height=3072, uneven=1, bins=64,
             fields="8/32/128", src="f32", dst="f32"),
        # one training step on one small crop, through the autograd function
        dict(name="train-512x384", kind="autograd", images=1, width=512, height=384, bins=32, fields="4/16/64"),
        # one training step on a batch of 16 one-megapixel crops: forward, input and parameter gradients
        dict(name="train-16x1024", kind="train", images=16, width=1024, height=1024, bins=32, fields="8/32/128"),
        # the gradient alone for a half-precision image of odd size (the forward is recomputed)
        dict(name="gradient-1599x1199-f16", kind="gradient", images=1, width=1599, height=1199, bins=32,
             fields="8/32/128", src="f16"),
        # the integral histogram itself, handed to another method
        dict(name="histogram-1080p", kind="histogram", width=1920, height=1080, bins=32),
        # the capture front-end: four bracketed 12 MP exposures into a radiance map
        dict(name="merge-4x12mp", kind="merge", images=4, width=4000, height=3000, dst="f32"),
    ]


def _size(rng, lo, hi):
    """A width log-uniform in lo..hi and a height of 0.5 to 1 times it, odd ones among them."""
    w = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return w, max(1, int(round(w * rng.uniform(0.5, 1.0))))


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "forward", "batch", "autograd", "train", "gradient",
                       "histogram", "merge"])
    bins = int(round(math.exp(rng.uniform(math.log(5), math.log(64)))))
    fields = rng.choice(["4/16/64", "8/32/128", "8/32/128", "5/40", "3/12/48/96"])
    if kind == "forward":
        w, h = _size(rng, 320, 4096)
        if rng.random() < 0.25:
            fields, bins = "pyramid%d" % rng.randint(3, 5), rng.randint(4, 12)
        return dict(kind=kind, width=w, height=h, bins=bins, fields=fields, src=rng.choice(["f32", "f32", "f16"]),
                    dst=rng.choice(["f32", "f32", "f16", "u8"]))
    if kind == "batch":
        if rng.random() < 0.5:
            w, h = _size(rng, 640, 1920)
            return dict(kind=kind, images=rng.randint(2, 60), width=w, height=h, uneven=0, bins=bins, fields=fields,
                        src="f16", dst="f16")
        return dict(kind=kind, images=rng.randint(3, 16), width=4096, height=3072, uneven=rng.randint(2, 9999),
                    bins=bins, fields=fields, src="f32", dst="f32")
    if kind == "autograd":
        w, h = _size(rng, 256, 1024)
        return dict(kind=kind, images=rng.randint(1, 3), width=w, height=h, bins=bins, fields=fields)
    if kind == "train":
        w, h = _size(rng, 256, 1200)
        return dict(kind=kind, images=rng.randint(2, 16), width=w, height=h, bins=bins, fields=fields)
    if kind == "gradient":
        w, h = _size(rng, 320, 2400)
        return dict(kind=kind, images=1, width=w, height=h, bins=bins, fields=fields, src=rng.choice(["f32", "f16"]))
    w, h = _size(rng, 320, 2048) if kind == "histogram" else _size(rng, 640, 4096)
    if kind == "histogram":
        return dict(kind=kind, width=w, height=h, bins=bins)
    return dict(kind=kind, images=rng.randint(2, 6), width=w, height=h, dst=rng.choice(["f32", "f16"]))


def _sizes(case):
    """(height, width) of each image of the case."""
    n = case.get("images", 1) if case["kind"] != "merge" else 1
    if not case.get("uneven"):
        return [(case["height"], case["width"])] * n
    rng, out = np.random.default_rng(case["uneven"]), []  # widths 640.., aspect 4:3 or 16:9, heights 480..
    while len(out) < n:
        w = int(rng.integers(640, case["width"] + 1))
        h = int(round(w / (4 / 3 if rng.uniform() < 0.5 else 16 / 9)))
        if 480 <= h <= case["height"]:
            out.append((h, w))
    return out


def _pixels(case):
    return sum(h * w for h, w in _sizes(case))


def _radii(case):
    """Half-sizes (rx, ry) of the case's fields."""
    f = case["fields"]
    if f.startswith("pyramid"):
        return [(case["width"] >> (i + 1), case["height"] >> (i + 1)) for i in range(int(f[7:]))]
    return [(int(r), int(r)) for r in f.split("/")]


# ------------------------------------------------------------------ inputs --
def _scenes(n, h, w, seed, dtype):
    """n wide-dynamic-range scenes (n, h, w, 3): a luminance ramp over six decades in a random direction, 20
    rectangles half to two decades brighter or darker with a chroma of their own, 2 % noise per pixel."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    out = torch.empty((n, h, w, 3), dtype=dtype, device="cuda")
    yy = torch.linspace(-0.5, 0.5, h, device="cuda")[:, None]
    xx = torch.linspace(-0.5, 0.5, w, device="cuda")[None, :]
    rects = None
    for i in range(n):
        if i % 30 == 0:  # a new scene; the images between are its next frames
            theta = rng.uniform(0, 2 * math.pi)
            a, b = math.cos(theta), math.sin(theta)
            lo = -(abs(a) + abs(b)) / 2
            ramp = (a * xx + b * yy - lo) / max(-2 * lo, 1e-12)
            rects = [(rng.uniform(), rng.uniform(), rng.uniform(0.03, 0.3), rng.uniform(0.03, 0.3),
                      rng.uniform(0.5, 2.0) * rng.choice([-1.0, 1.0]), rng.uniform(0.2, 0.8, 3),
                      rng.uniform(-3, 3, 2)) for _ in range(20)]
            back = rng.uniform(0.2, 0.8, 3)
        t = i % 30
        dec = -2.0 + 6.0 * ramp + 0.01 * t
        chroma = [torch.full((h, w), float(back[c] / back.mean()), device="cuda") for c in range(3)]
        for fy, fx, rh, rw, amp, col, v in rects:
            bh, bw = max(1, int(rh * h)), max(1, int(rw * w))
            y0, x0 = int(fy * max(h - bh, 1) + v[0] * t) % h, int(fx * max(w - bw, 1) + v[1] * t) % w
            dec[y0:y0 + bh, x0:x0 + bw] += amp
            for c in range(3):
                chroma[c][y0:y0 + bh, x0:x0 + bw] = float(col[c] / col.mean())
        lum = torch.pow(10.0, dec.clamp_(-2.0, 4.0))
        lum *= 1.0 + 0.02 * torch.randn((h, w), generator=gen, device="cuda")
        lum.clamp_(min=1e-5)
        for c in range(3):
            out[i, :, :, c] = lum * chroma[c]
    return out


@functools.lru_cache(maxsize=3)
def _mapper(bins, radii, reuse):
    """The context a program keeps for all its images of one setting."""
    m = tm.ToneMapper(tm.make_params(bins, list(radii)))
    if reuse:
        tm.tm_set_option(m.ctx, tm.TM_OPT_BACKWARD_REUSE, 1)
    return m


@functools.lru_cache(maxsize=3)
def _autograd_cache(bins, radii):
    return tm._CtxCache(tm.make_params(bins, list(radii)))


TIMES = [1.0 / 1024, 1.0 / 128, 1.0 / 16, 0.5, 4.0, 32.0]  # a bracket, three stops apart


def _log_response():
    """g(z) = ln of the sensor exposure that a power-law camera maps to z, per channel."""
    z = np.arange(256, dtype=np.float64)
    z[0] = 1.0
    return np.repeat((2.2 * np.log(z / 255.0))[None, :], 3, axis=0)


def prepare(case, seed):
    kind, sizes = case["kind"], _sizes(case)
    state = {"case": case}
    if kind == "histogram":
        x = _scenes(1, *sizes[0], seed, torch.float32)[0]
        lum = torch.log(x.mean(2))
        lum = (lum - lum.min()) / (lum.max() - lum.min())
        state["bins"] = (lum * case["bins"]).clamp(0, case["bins"] - 1).to(torch.uint8)
        h, w = sizes[0]
        state["planes"] = torch.empty((case["bins"], h + 1, w + 1), dtype=torch.int32, device="cuda")
        return state
    if kind == "merge":
        x = _scenes(1, *sizes[0], seed, torch.float32)[0]
        state["times"] = TIMES[:case["images"]]
        state["ldr"] = [(255.0 * (x * t).clamp(0, 1) ** (1 / 2.2)).round().to(torch.uint8) for t in state["times"]]
        state["response"] = _log_response()
        state["y"] = torch.empty(x.shape, dtype=DTYPES[case["dst"]], device="cuda")
        return state
    src = DTYPES[case.get("src", "f32")]
    if case.get("uneven"):
        xs = [_scenes(1, h, w, seed + 1000 * i, src)[0] for i, (h, w) in enumerate(sizes)]
        state["x"], state["xs"] = xs, xs
        state["y"] = [torch.empty(x.shape, dtype=DTYPES[case["dst"]], device="cuda") for x in xs]
        state["ys"] = state["y"]
    else:
        state["x"] = _scenes(len(sizes), *sizes[0], seed, src)
        state["xs"] = list(state["x"])
        if "dst" in case or kind == "train":
            state["y"] = torch.empty(state["x"].shape, dtype=DTYPES[case.get("dst", "f32")], device="cuda")
            state["ys"] = list(state["y"])
    if kind in ("autograd", "train", "gradient"):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) + 77)
        state["g"] = torch.randn(state["x"].shape, generator=gen, device="cuda")
        state["gs"] = list(state["g"])
    radii = tuple(_radii(case))
    if kind == "autograd":
        state["cache"] = _autograd_cache(case["bins"], radii)
        state["theta"] = tm.params_tensor(state["cache"].template).requires_grad_(True)
        state["x"] = (state["x"][0] if case["images"] == 1 else state["x"]).requires_grad_(True)
        state["g"] = state["g"][0] if case["images"] == 1 else state["g"]
        return state
    state["mapper"] = _mapper(case["bins"], radii, kind == "train")
    if kind in ("train", "gradient"):
        state["gx"] = torch.empty(state["x"].shape, dtype=torch.float32, device="cuda")
        state["gxs"] = list(state["gx"])
        state["gp"] = torch.empty(3 + 2 * len(radii), dtype=torch.float32, device="cuda")
    return state


# -------------------------------------------------------------------- runs --
def run(state):
    kind = state["case"]["kind"]
    if kind == "histogram":
        tm.tm_integral_histogram(state["bins"], state["case"]["bins"], state["planes"])
        return state["planes"]
    if kind == "merge":
        tm.tm_merge_exposures(state["ldr"], state["times"], state["response"], state["y"])
        return state["y"]
    if kind == "autograd":
        y = tm.TMFunction.apply(state["x"], state["theta"], state["cache"])
        gx, gp = torch.autograd.grad(y, (state["x"], state["theta"]), state["g"])
        return {"y": y.detach(), "gx": gx, "gp": gp}
    ctx = state["mapper"].ctx
    if kind == "forward":
        tm.tm_forward(ctx, state["xs"][0], state["ys"][0])
        return state["ys"][0]
    if kind == "batch":
        tm.tm_forward_batch(ctx, state["xs"], state["ys"])
        return state["y"]
    if kind == "train":
        tm.tm_forward_batch(ctx, state["xs"], state["ys"])
        tm.tm_backward_batch(ctx, state["xs"], state["gs"], state["gxs"], state["gp"])
        return {"y": state["y"], "gx": state["gx"], "gp": state["gp"]}
    tm.tm_backward(ctx, state["xs"][0], state["gs"][0], state["gxs"][0], state["gp"])
    return {"gx": state["gx"], "gp": state["gp"]}


def work(case):
    n, kind = _pixels(case), case["kind"]
    if kind == "histogram":
        h, w = _sizes(case)[0]
        return {"bytes": n + 4 * case["bins"] * (h + 1) * (w + 1), "flops": 2 * case["bins"] * n}
    size = {"f32": 12, "f16": 6, "u8": 3}  # bytes of a pixel
    if kind == "merge":
        return {"bytes": n * (3 * case["images"] + size[case["dst"]]), "flops": n * 3 * (4 * case["images"] + 10)}
    s = len(_radii(case))
    if kind in ("forward", "batch"):
        return {"bytes": n * (size[case["src"]] + size[case["dst"]]), "flops": n * (60 + 50 * s)}
    out = 12 if kind != "gradient" else 0
    return {"bytes": n * (size[case.get("src", "f32")] + 12 + 12 + out), "flops": n * (150 + 150 * s)}


# ------------------------------------------------------------ 64-bit values --
def _box(v, rx, ry):
    """Sums of v (h, w), 64-bit, over the windows [x - rx, x + rx] x [y - ry, y + ry] clipped to the image."""
    h, w = v.shape
    rx, ry = min(rx, w - 1), min(ry, h - 1)
    if max(rx, ry) <= 200:  # summed directly: no cancellation in small windows
        for r, k in ((rx, (1, 2 * rx + 1)), (ry, (2 * ry + 1, 1))):
            v = torch.nn.functional.avg_pool2d(v[None, None], k, 1, (0, r) if k[0] == 1 else (r, 0),
                                               divisor_override=1)[0, 0]
        return v
    c = torch.nn.functional.pad(v.cumsum(0).cumsum(1), (1, 0, 1, 0))
    x, y = torch.arange(w, device=v.device), torch.arange(h, device=v.device)
    x0, x1 = (x - rx).clamp(min=0), (x + rx + 1).clamp(max=w)
    y0, y1 = (y - ry).clamp(min=0), (y + ry + 1).clamp(max=h)
    c = c[y1] - c[y0]
    return c[:, x1] - c[:, x0]


def _area(h, w, rx, ry):
    x, y = torch.arange(w, device="cuda"), torch.arange(h, device="cuda")
    nx = (x + rx).clamp(max=w - 1) - (x - rx).clamp(min=0) + 1
    ny = (y + ry).clamp(max=h - 1) - (y - ry).clamp(min=0) + 1
    return (ny[:, None] * nx[None, :]).double()


def _counts(b, bins, radii):
    """For every field, how many pixels of each pixel's window have a smaller bin than it."""
    h, w = b.shape
    out = [torch.zeros((h, w), dtype=torch.float64, device="cuda") for _ in radii]
    for k in range(1, bins):
        ys, xs = (b == k).nonzero(as_tuple=True)
        if not ys.numel():
            continue
        c = torch.nn.functional.pad((b < k).to(torch.int32).cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32),
                                    (1, 0, 1, 0))
        for f, (rx, ry) in enumerate(radii):
            x0, x1 = (xs - rx).clamp(min=0), (xs + rx + 1).clamp(max=w)
            y0, y1 = (ys - ry).clamp(min=0), (ys + ry + 1).clamp(max=h)
            out[f][ys, xs] = (c[y1, x1] - c[y0, x1] - c[y1, x0] + c[y0, x0]).double()
    return out


def _tone_map(x, theta, bins, radii):
    """The operator on one image x (h, w, 3), 64-bit, theta = [ld_min, ld_max, sat, eps..., alpha...]. The
    luminance that is binned is the float32 one, as the operator defines it; the bins are held fixed."""
    h, w, _ = x.shape
    s = len(radii)
    f = x.detach().float()
    l32 = (0.2126 * f[..., 0] + 0.7152 * f[..., 1]) + 0.0722 * f[..., 2]
    l32 = l32.clamp(min=float(np.float32(1e-30))).double()
    lum = 0.2126 * x[..., 0] + 0.7152 * x[..., 1] + 0.0722 * x[..., 2]
    lum = l32 + (lum - lum.detach())
    flat = lum.reshape(-1)
    lo = torch.log(flat[(l32.reshape(-1) == l32.min()).nonzero()[0, 0]])
    hi = torch.log(flat[(l32.reshape(-1) == l32.max()).nonzero()[0, 0]])
    lhat = (torch.log(lum) - lo) / (hi - lo)
    k = torch.arange(1, bins, dtype=torch.float64, device="cuda")
    edges = torch.exp(lo.detach() + (hi - lo).detach() * (k / bins))
    b = torch.bucketize(l32, edges, right=True)
    top, fused, plain = 0.0, 0.0, 0.0
    for i, cnt in enumerate(_counts(b, bins, radii)):
        n = _area(h, w, *radii[i])
        m = _box(lhat - 0.5, *radii[i]) / n
        var = (_box((lhat - 0.5) ** 2, *radii[i]) / n - m * m).clamp(min=0)
        lf = theta[0] + (theta[1] - theta[0]) * (cnt / n)
        wf = theta[3 + s + i] * var / (var + theta[3 + i])
        top, fused, plain = top + wf, fused + wf * lf, plain + lf / s
    tone = torch.where(top > 0, fused / torch.where(top > 0, top, torch.ones_like(top)), plain)
    rho = (x / lum[..., None]).clamp(min=0)
    return torch.pow(rho, theta[2]) * tone[..., None]


def _theta(s):
    return torch.tensor([0.0, 1.0, SAT] + [EPS] * s + [1.0] * s, dtype=torch.float64, device="cuda")


def exact(case, seed):
    kind = case["kind"]
    if kind == "histogram" or case.get("dst") == "u8":
        return None  # whole numbers
    state = prepare(case, seed)
    if kind == "merge":
        g = torch.tensor(state["response"], dtype=torch.float32, device="cuda").double()
        num = den = 0.0
        for z, t in zip(state["ldr"], state["times"]):
            zi = z.long()
            wt = torch.where(zi <= 127, zi, 255 - zi).double()
            gz = torch.stack([g[c][zi[..., c]] for c in range(3)], dim=-1)
            num, den = num + wt * (gz - math.log(t)), den + wt
        short, long_ = int(np.argmin(state["times"])), int(np.argmax(state["times"]))
        at = torch.where(state["ldr"][short] == 255, state["ldr"][short], state["ldr"][long_]).long()
        ln_t = torch.where(state["ldr"][short] == 255, math.log(state["times"][short]), math.log(state["times"][long_]))
        only = torch.stack([g[c][at[..., c]] for c in range(3)], dim=-1) - ln_t
        return torch.exp(torch.where(den > 0, num / den.clamp(min=1.0), only))
    radii, bins = _radii(case), case["bins"]
    theta = _theta(len(radii))
    if kind in ("forward", "batch"):
        ys = [_tone_map(x.double(), theta, bins, radii) for x in state["xs"]]
        return ys[0] if kind == "forward" else ys if case["uneven"] else torch.stack(ys)
    ys, gxs, gp = [], [], torch.zeros_like(theta)
    for x, g in zip(state["xs"], state["gs"]):
        x, th = x.detach().double().requires_grad_(True), theta.clone().requires_grad_(True)
        y = _tone_map(x, th, bins, radii)
        gx, gt = torch.autograd.grad(y, (x, th), g.double())
        ys.append(y.detach())
        gxs.append(gx)
        gp += gt
    gx, y = torch.stack(gxs), torch.stack(ys)
    if kind == "autograd":
        one = case["images"] == 1
        return {"y": y[0] if one else y, "gx": gx[0] if one else gx, "gp": gp}
    return {"y": y, "gx": gx, "gp": gp} if kind == "train" else {"gx": gx, "gp": gp}
