"""The work a user of this package gives it, as cases that can be timed and compared.

An ABCD program spends its time in a handful of calls: the active-block training step, the
refresh of a block's cached layers, the folds of cached layers into F and B (dense, packed and
in pieces), the layers' visibility, and the evaluation of a full composite.  The listed cases
take each of them through the package's public entry points at the sizes of this repository's
workloads (the tiny, 3x3x3 and scene-scale grids, the 64-layer compositing sweep, the
2M-Gaussian stress block) and at odd, ragged ones; `draw` spreads the same kinds over the range
in between.

Inputs are drawn on the GPU from the seed with the distributions of the package's synthetic
scenes (means uniform in a grid cell or from a 16-blob mixture, log-scales N(log(0.05 side), 0.5),
random rotations, logits N(0, 1)), seen by a camera at a random place of the ring around the
grid.  `exact` recomputes every result with plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2608_27735_gb300 as ab
from paper_2608_27735_gb300.bcd import default_lr

DEV = "cuda"
SIDE = 5.0
LAM = 0.2
BETA1, BETA2, EPS = 0.9, 0.999, 1e-15
STEP0 = 250                       # a step in the middle of a stage of T = 500
# a late stage's rates, a hundredth of the defaults: the block hardly moves while it is timed
LR_SCALE = 0.01
NEAR, DILATION, GUARD, ALPHA_MAX, ALPHA_MIN, T_MIN = 0.2, 0.3, 1.3, 0.99, 1.0 / 255.0, 1e-4


# ---------------------------------------------------------------------------------------
# the cases

def listed():
    return [
        # one active-block training step (render, composite with F and B, loss, backward, Adam)
        # of the tiny grid: latency and launches
        {"name": "step_2k_128", "kind": "step", "n": 2000, "sh": 0, "w": 128, "h": 128,
         "grid": "2x2x2", "fb": "f16", "bg": False},
        # the same step on the 3x3x3 grid's centre block
        {"name": "step_20k_640x480", "kind": "step", "n": 20000, "sh": 3, "w": 640, "h": 480,
         "grid": "3x3x3", "fb": "f16", "bg": False},
        # odd sizes, ragged tiles on both axes, 32-bit F and B, a background colour
        {"name": "step_33k_1001x667", "kind": "step", "n": 33333, "sh": 2, "w": 1001, "h": 667,
         "grid": "3x2x2", "fb": "f32", "bg": True},
        # the step the headline benchmark repeats: one block of the 4x4x2 grid
        {"name": "step_100k_1237x822", "kind": "step", "n": 100000, "sh": 3, "w": 1237, "h": 822,
         "grid": "4x4x2", "fb": "f16", "bg": False},
        # forward and backward of the stress block: dense tiles, deep overlap, the largest call
        {"name": "grad_2M_1920x1080", "kind": "grad", "n": 2000000, "sh": 3, "w": 1920, "h": 1080,
         "grid": "mixture", "fb": "none", "bg": False},
        # one camera's cached layer of a block rendered again at a stage's end (packed form)
        {"name": "refresh_packed_100k", "kind": "refresh_packed", "n": 100000, "sh": 3, "w": 1237,
         "h": 822, "grid": "4x4x2"},
        # the same into a dense fp16 layer, as the block coordinate descent driver does
        {"name": "refresh_dense_20k", "kind": "refresh_dense", "n": 20000, "sh": 3, "w": 640,
         "h": 480, "grid": "3x3x3"},
        # F and B of one camera from 64 dense layers (the compositing sweep)
        {"name": "composite_64_1080p", "kind": "composite", "layers": 64, "w": 1920, "h": 1080,
         "dtype": "f16"},
        # F and B from the packed layers of the 4x4x2 grid, at the start of a stage
        {"name": "composite_packed_32", "kind": "composite_packed", "layers": 32, "w": 1237,
         "h": 822, "fill": 0.33},
        # visible share and coverage of the same layers (culling of camera-block pairs)
        {"name": "visibility_packed_32", "kind": "visibility_packed", "layers": 32, "w": 1237,
         "h": 822, "fill": 0.33},
        # evaluation: the full composite of a camera's layers and its loss, without a gradient
        {"name": "eval_27_640x480", "kind": "eval", "layers": 27, "w": 640, "h": 480},
        # the out-of-core driver's fold of one side in pieces that fit its staging buffer
        {"name": "fold_packed_31_1001x667", "kind": "fold_packed", "layers": 31, "w": 1001,
         "h": 667, "fill": 0.4, "piece": 8},
    ]


def _odd(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "grad", "refresh_packed", "refresh_dense", "composite",
                       "composite_packed", "visibility_packed", "eval", "fold_packed"])
    w = _odd(rng, 100, 1920)
    h = max(64, min(1200, int(w * rng.uniform(0.5, 1.0))))
    c = {"kind": kind, "w": w, "h": h}
    if kind in ("step", "grad", "refresh_packed", "refresh_dense"):
        c["grid"] = rng.choice(["2x2x2", "3x3x3", "3x2x2", "4x4x2", "mixture"])
        c["n"] = _odd(rng, 1000, 300000)
        c["sh"] = rng.choice([0, 1, 2, 3, 3])
        if kind in ("step", "grad"):
            c["fb"] = rng.choice(["f16", "f16", "f32", "none"])
            c["bg"] = rng.random() < 0.3
    else:
        c["layers"] = _odd(rng, 2, 64)
        if kind == "composite":
            c["dtype"] = rng.choice(["f16", "f16", "f32"])
        if kind in ("composite_packed", "visibility_packed", "fold_packed"):
            c["fill"] = round(rng.uniform(0.1, 0.9), 2)
        if kind == "fold_packed":
            c["piece"] = rng.randint(1, c["layers"])
    return c


# ---------------------------------------------------------------------------------------
# inputs (plain tensors, from the seed alone)

class Cam:
    """A pinhole camera as the package's camera() reads it."""

    def __init__(self, pos, w, h, fov=60.0):
        p = np.asarray(pos, np.float64)
        f = -p / np.linalg.norm(p)
        r = np.cross(f, np.array([0.0, 0.0, 1.0]))
        r /= np.linalg.norm(r)
        d = np.cross(f, r)
        self.R = np.stack([r, d, f]).astype(np.float32)
        self.t = (-self.R.astype(np.float64) @ p).astype(np.float32)
        self.fx = self.fy = float(np.float32(0.5 * w / math.tan(math.radians(fov) / 2.0)))
        self.cx, self.cy = float(np.float32(w / 2.0)), float(np.float32(h / 2.0))
        self.width, self.height = int(w), int(h)


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 64 + stream)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _half_diag(dims):
    return 0.5 * SIDE * math.sqrt(sum(d * d for d in dims))


def _dims(case):
    return (4, 4, 4) if case["grid"] == "mixture" else tuple(int(v) for v in case["grid"].split("x"))


def _block(case, seed):
    """The active block's parameters (means, log-scales, quaternions, logits, SH) and the
    camera: a cell near the grid's middle, or the mixture, and a ring camera."""
    g = _gen(seed, 1)
    n, D = case["n"], (case["sh"] + 1) ** 2
    rng = np.random.default_rng(int(seed) * 64 + 2)
    if case["grid"] == "mixture":
        centres = 20.0 * (_rand(g, 16, 3) - 0.5)
        means = centres[torch.randint(16, (n,), generator=g, device=DEV)] + _randn(g, n, 3)
        radius, jitter = 30.0, 2.0
    else:
        dims = _dims(case)
        lo = torch.tensor([SIDE * ((d - 1) // 2 - 0.5 * d) for d in dims], device=DEV)
        means = lo + SIDE * (0.0001 + 0.9998 * _rand(g, n, 3))
        radius, jitter = 1.5 * _half_diag(dims), 0.1 * SIDE * dims[2]
    a = rng.uniform(0.0, 2.0 * math.pi)
    cam = Cam((radius * math.cos(a), radius * math.sin(a), rng.uniform(-jitter, jitter)), case["w"], case["h"])
    ls = math.log(0.05 * SIDE) + 0.5 * _randn(g, n, 3)
    q = torch.nn.functional.normalize(_randn(g, n, 4), dim=1)
    logits = _randn(g, n)
    sh = 0.05 * _randn(g, n, D, 3)
    sh[:, 0] = math.sqrt(math.pi) * (2.0 * _rand(g, n, 3) - 1.0)
    return [t.contiguous() for t in (means, ls, q, logits, sh)], cam


def _smooth(g, h, w, ch, cell=48):
    x = _rand(g, 1, ch, max(2, h // cell + 2), max(2, w // cell + 2))
    return torch.nn.functional.interpolate(x, size=(h, w), mode="bilinear", align_corners=True)[0].permute(1, 2, 0)


def _images(case, seed):
    """F, B (premultiplied RGBA, or None) and the target of one camera."""
    g = _gen(seed, 3)
    h, w = case["h"], case["w"]
    gt = (0.8 * _smooth(g, h, w, 3) + 0.2 * _rand(g, h, w, 3)).contiguous()
    if case["fb"] == "none":
        return None, None, gt
    dt = torch.float16 if case["fb"] == "f16" else torch.float32
    out = []
    for gain, off in ((1.6, -0.7), (1.6, -0.2)):           # F is mostly clear, B mostly covered
        a = (gain * _smooth(g, h, w, 1) + off).clamp(0.0, 0.98)
        out.append(torch.cat([a * _smooth(g, h, w, 3), a], -1).to(dt).contiguous())
    return out[0], out[1], gt


def _bg(case):
    return (0.2, 0.5, 0.7) if case.get("bg") else None


def _moments(params, seed):
    """Adam moments as a running stage leaves them."""
    g = _gen(seed, 4)
    m = [1e-6 * _randn(g, *t.shape) for t in params]
    v = [(1e-5 * _rand(g, *t.shape)).square() for t in params]
    return m, v


def _lr(case):
    dims = _dims(case)
    return [LR_SCALE * x for x in default_lr(2.0 * _half_diag(dims))]


def _dense_layers(case, seed, dtype):
    g = _gen(seed, 5)
    out = []
    for _ in range(case["layers"]):
        a = _rand(g, case["h"], case["w"], 1)
        out.append(torch.cat([a * _rand(g, case["h"], case["w"], 3), a], -1).to(dtype))
    return out


def _order(case, seed):
    rng = np.random.default_rng(int(seed) * 64 + 6)
    L = case["layers"]
    return [int(k) for k in rng.permutation(L)], int(rng.integers(0, L))


def _packed_layers(case, seed):
    """Per layer a tile map over the 16x16 tiles (-1: clear) and its stored tiles: a block's
    footprint, an ellipse of tiles around a random centre."""
    g = _gen(seed, 7)
    tx, ty = (case["w"] + 15) // 16, (case["h"] + 15) // 16
    ys, xs = torch.meshgrid(torch.arange(ty, device=DEV), torch.arange(tx, device=DEV), indexing="ij")
    maps, data = [], []
    for _ in range(case["layers"]):
        cx, cy = (0.25 + 0.5 * _rand(g, 2)).unbind()
        r = ((xs + 0.5) / tx - cx) ** 2 + ((ys + 0.5) / ty - cy) ** 2
        stored = (r <= torch.quantile(r.flatten().float(), case["fill"])).flatten()
        idx = torch.cumsum(stored.int(), 0, dtype=torch.int32) - 1
        maps.append(torch.where(stored, idx, torch.full_like(idx, -1)).contiguous())
        k = max(1, int(stored.sum()))
        a = _rand(g, k, 16, 16, 1).square()
        data.append(torch.cat([a * _rand(g, k, 16, 16, 3), a], -1).half().contiguous())
    return maps, data


# ---------------------------------------------------------------------------------------
# what a user's program holds, and one pass

def _gauss(arrays, sh):
    return ab.Gaussians(*arrays, sh)


def _block_state(case, seed):
    """The block on the device, a context with its workspace, and the projection and list
    buffers sized once from the block's tile rectangles."""
    params, cam_np = _block(case, seed)
    n, w, h = case["n"], case["w"], case["h"]
    s = {"case": case, "theta": _gauss(params, case["sh"]), "cam": ab.camera(cam_np), "ctx": ab.Context(0)}
    s["proj"] = ab.Projected.alloc(n)
    ab.abcd_project(s["ctx"], s["theta"], s["cam"], None, s["proj"])
    cap = int(1.3 * int(s["proj"].tiles_touched.sum(dtype=torch.int64))) + 4096
    s["ctx"].reserve(n, cap, w * h)
    s["tiles"] = ab.Tiles.alloc(cap, w, h)
    return s


def prepare(case, seed):
    kind, w, h = case["kind"], case["w"], case["h"]
    if kind in ("step", "grad"):
        s = _block_state(case, seed)
        s["F"], s["B"], s["gt"] = _images(case, seed)
        s["fbd"] = ab.ABCD_F32 if case["fb"] == "f32" else ab.ABCD_F16
        s["out"] = torch.zeros(h, w, 4, device=DEV)
        s["fwd"] = ab.FwdState.alloc(w, h)
        s["loss"] = torch.zeros(1, device=DEV)
        s["grads"] = ab.Gaussians.zeros_like(s["theta"])
        if kind == "step":
            m, v = _moments(s["theta"].tensors(), seed)
            s["m"], s["v"] = _gauss(m, case["sh"]), _gauss(v, case["sh"])
            s["call"] = ab.TrainStep(s["ctx"], s["theta"], s["grads"], s["m"], s["v"], s["proj"], s["tiles"],
                                     s["out"], s["fwd"], _lr(case), BETA1, BETA2, EPS, LAM, bg=_bg(case))
            s["t"] = STEP0
        return s
    if kind == "refresh_packed":
        s = _block_state(case, seed)
        nt = ((w + 15) // 16) * ((h + 15) // 16)
        s["map"] = torch.zeros(nt, dtype=torch.int32, device=DEV)
        s["packed"] = torch.zeros(nt, 16, 16, 4, dtype=torch.float16, device=DEV)
        s["count"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        s["call"] = ab.RefreshLayer(s["ctx"], s["theta"], s["proj"], s["tiles"])
        return s
    if kind == "refresh_dense":
        s = _block_state(case, seed)
        s["layer"] = torch.zeros(h, w, 4, dtype=torch.float16, device=DEV)
        return s
    s = {"case": case, "ctx": ab.Context(0)}
    if kind in ("composite", "eval"):
        dt = torch.float32 if case.get("dtype") == "f32" else torch.float16
        s["layers"] = _dense_layers(case, seed, dt)
        s["order"], s["split"] = _order(case, seed)
    else:
        s["maps"], s["data"] = _packed_layers(case, seed)
        s["order"], s["split"] = _order(case, seed)
    if kind in ("composite", "composite_packed"):
        s["F"] = torch.zeros(h, w, 4, dtype=torch.float16, device=DEV)
        s["B"] = torch.zeros_like(s["F"])
    if kind == "composite_packed":
        s["tables"] = ab.PackedLayers(s["maps"], s["data"], s["order"], s["split"])
    if kind == "visibility_packed":
        s["ctx"].reserve(1024, 1024, w * h)
        s["tables"] = ab.PackedLayers(s["maps"], s["data"], s["order"], case["layers"])
        s["visible"] = torch.zeros(case["layers"], dtype=torch.float64, device=DEV)
        s["coverage"] = torch.zeros_like(s["visible"])
    if kind == "eval":
        s["ctx"].reserve(1024, 1024, w * h)
        s["gt"] = _images({**case, "fb": "none"}, seed)[2]
        s["full"] = torch.zeros(h, w, 4, device=DEV)
        s["loss"] = torch.zeros(1, device=DEV)
    if kind == "fold_packed":
        s["acc"] = torch.zeros(h, w, 4, device=DEV)
        s["out16"] = torch.zeros(h, w, 4, dtype=torch.float16, device=DEV)
    return s


def run(s):
    case = s["case"]
    kind, w, h = case["kind"], case["w"], case["h"]
    ctx = s["ctx"]
    if kind == "step":
        s["t"] += 1
        s["call"](s["cam"], s["F"], s["B"], s["gt"], s["loss"], s["t"], s["fbd"])
        return {"out": s["out"], "loss": s["loss"], "grads": list(s["grads"].tensors()),
                "theta": list(s["theta"].tensors()), "m": list(s["m"].tensors()), "v": list(s["v"].tensors())}
    if kind == "grad":
        bg = _bg(case)
        ab.abcd_project(ctx, s["theta"], s["cam"], None, s["proj"])
        ab.abcd_bin_sort(ctx, s["proj"], case["n"], s["cam"], s["tiles"])
        ab.abcd_render_composite_fwd(ctx, s["cam"], None, s["proj"], s["tiles"], s["F"], s["B"], s["fbd"], bg,
                                     s["out"], s["fwd"])
        ab.abcd_backward(ctx, s["theta"], s["cam"], None, s["proj"], s["tiles"], s["F"], s["B"], s["fbd"], bg,
                         s["out"], s["fwd"], s["gt"], LAM, s["loss"], None, s["grads"])
        return {"out": s["out"], "loss": s["loss"], "grads": list(s["grads"].tensors())}
    if kind == "refresh_packed":
        s["call"](s["cam"], s["map"], s["packed"], s["count"])
        return {"map": s["map"], "packed": s["packed"], "count": s["count"]}
    if kind == "refresh_dense":
        ab.abcd_project(ctx, s["theta"], s["cam"], None, s["proj"])
        ab.abcd_bin_sort(ctx, s["proj"], case["n"], s["cam"], s["tiles"])
        ab.abcd_render_composite_fwd(ctx, s["cam"], None, s["proj"], s["tiles"], refresh_f16=s["layer"])
        return s["layer"]
    if kind == "composite":
        dt = ab.ABCD_F32 if case["dtype"] == "f32" else ab.ABCD_F16
        ab.abcd_composite_cache(ctx, s["layers"], s["order"], s["split"], w, h, s["F"], s["B"], dt)
        return [s["F"], s["B"]]
    if kind == "composite_packed":
        ab.abcd_composite_cache_packed_tables(ctx, s["tables"], w, h, s["F"], s["B"])
        return [s["F"], s["B"]]
    if kind == "visibility_packed":
        ab.abcd_layer_visibility_tables(ctx, s["tables"], w, h, s["visible"], s["coverage"])
        return [s["visible"], s["coverage"]]
    if kind == "eval":
        ab.abcd_composite_cache(ctx, s["layers"], s["order"], case["layers"], w, h, s["full"], None,
                                ab.ABCD_F16, ab.ABCD_F32)
        ab.abcd_loss(ctx, s["full"], s["gt"], w, h, LAM, s["loss"], None)
        return [s["full"], s["loss"]]
    # fold_packed: the pieces in order, the accumulator carried in 32 bits, rounded at the end
    L, p = case["layers"], case["piece"]
    for k in range(0, L, p):
        part = s["order"][k:k + p]
        ab.abcd_composite_fold_packed(ctx, [s["maps"][i] for i in part], [s["data"][i] for i in part], w, h,
                                      s["acc"] if k else None, s["acc"], s["out16"] if k + p >= L else None)
    return [s["acc"], s["out16"]]


# ---------------------------------------------------------------------------------------
# what a pass cannot do without

def _splat_work(case):
    """(pixels covered by a block's image, list positions walked over all pixels), from the
    geometry: a splat reaches alpha_min on about 27 sigma^2 pixels, and a pixel stops after about
    40 contributing layers."""
    w, h, n = case["w"], case["h"], case["n"]
    f = 0.5 * w / math.tan(math.radians(30.0))
    radius = 30.0 if case["grid"] == "mixture" else 1.5 * _half_diag(_dims(case))
    px = f * 0.05 * SIDE / radius                         # a splat's sigma in pixels
    extent = f * (20.0 if case["grid"] == "mixture" else 1.4 * SIDE) / radius
    covered = min(w * h, extent * extent)
    return covered, min(n * 27.0 * (px * px + 0.3), 40.0 * covered)


def work(case):
    kind = case["kind"]
    w, h = case["w"], case["h"]
    px = w * h
    if kind in ("step", "grad", "refresh_packed", "refresh_dense"):
        n, D = case["n"], (case["sh"] + 1) ** 2
        p = 4 * (11 + 3 * D) * n                          # one copy of the parameters
        covered, walked = _splat_work(case)
        if kind.startswith("refresh"):
            out = 8 * (covered if kind == "refresh_packed" else px)
            return {"bytes": p + out, "flops": 26.0 * walked + 400.0 * n}
        fb = {"f16": 16, "f32": 32, "none": 0}[case["fb"]]
        bytes_ = p * (7 if kind == "step" else 2) + px * (fb + 12 + 16)
        # blend 25 + exp, its backward 68 + exp; the loss's eight separable 11-tap windows over
        # three channels; the projection and its backward
        return {"bytes": bytes_, "flops": 95.0 * walked + 3 * 400.0 * px + 1500.0 * n}
    L = case["layers"]
    if kind == "composite":
        per = 16 if case["dtype"] == "f32" else 8
        return {"bytes": (L - 1) * per * px + 16 * px, "flops": 8.0 * (L - 1) * px}
    if kind == "eval":
        return {"bytes": L * 8 * px + (16 + 12) * px, "flops": 8.0 * L * px + 3 * 250.0 * px}
    tiles = ((w + 15) // 16) * ((h + 15) // 16)
    stored = case["fill"] * tiles * 2048 * L
    if kind == "composite_packed":
        return {"bytes": stored * (L - 1) / L + 4 * tiles * (L - 1) + 16 * px, "flops": 8.0 * case["fill"] * L * px}
    if kind == "visibility_packed":
        return {"bytes": stored + 4 * tiles * L, "flops": 6.0 * case["fill"] * L * px}
    pieces = -(-L // case["piece"])
    return {"bytes": stored + 4 * tiles * L + px * (16 + 32 * (pieces - 1) + 8), "flops": 8.0 * case["fill"] * L * px}


def tolerance(case):
    """About four times the distance to `exact`.  The steps' gradients are off by up to 6e-5: a
    rounding of sigma, alpha or T moves a decision at a threshold (alpha_min, t_min) now and
    then, which "max" allows for at a single value.  fp16 results are off by their rounding."""
    kind = case["kind"]
    if kind in ("step", "grad"):
        return {"rel": 3e-4, "max": 0.5, "differ": 0.0}
    if kind.startswith("refresh"):
        return {"rel": 7e-4, "max": 0.05, "differ": 1e-3}
    if kind == "visibility_packed":
        return {"rel": 1e-7, "max": 1e-6}
    if kind == "eval":
        return {"rel": 1e-6}
    return {"rel": 7e-4, "max": 2e-3}


# ---------------------------------------------------------------------------------------
# the same results in 64 bits

def _f32(x):
    return float(np.float32(x))


def _sh_basis(deg, d):
    """Real spherical harmonics at unit directions d [n, 3] (Condon-Shortley phase), index
    l*l + l + m."""
    x, y, z = d.unbind(1)
    one = torch.ones_like(x)
    k = lambda l, m: math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
    leg = {(0, 0): one, (1, 0): z, (1, 1): one, (2, 0): 1.5 * z * z - 0.5, (2, 1): 3 * z, (2, 2): 3 * one,
           (3, 0): 2.5 * z ** 3 - 1.5 * z, (3, 1): 7.5 * z * z - 1.5, (3, 2): 15 * z, (3, 3): 15 * one}
    re, im = [one], [torch.zeros_like(x)]
    for _ in range(3):                                    # (x + i y)^m
        re.append(re[-1] * x - im[-1] * y)
        im.append(re[-2] * y + im[-1] * x)
    out = []
    for l in range(deg + 1):
        for m in range(-l, l + 1):
            a = abs(m)
            c = k(l, a) * (1.0 if m == 0 else math.sqrt(2.0) * (-1.0) ** a)
            out.append(c * leg[l, a] * (one if m == 0 else (re[a] if m > 0 else im[a])))
    return torch.stack(out, 1)


def _project64(params, cam, deg):
    """uv, conic (a, b, c), opacity, colour and radius of every Gaussian, differentiable."""
    mu, ls, q, logit, sh = params
    R = torch.tensor(cam.R, dtype=torch.float64, device=DEV)
    t = torch.tensor(cam.t, dtype=torch.float64, device=DEV)
    p = mu @ R.T + t
    z = p[:, 2]
    lim = torch.tensor([GUARD * 0.5 * cam.width / cam.fx, GUARD * 0.5 * cam.height / cam.fy],
                       dtype=torch.float64, device=DEV)
    xy = p[:, :2] / z[:, None]
    g = torch.minimum(torch.maximum(xy, -lim), lim) * z[:, None]
    zero = torch.zeros_like(z)
    J = torch.stack([torch.stack([cam.fx / z, zero, -cam.fx * g[:, 0] / (z * z)], 1),
                     torch.stack([zero, cam.fy / z, -cam.fy * g[:, 1] / (z * z)], 1)], 1)
    w, x, y, qz = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    Rq = torch.stack([1 - 2 * (y * y + qz * qz), 2 * (x * y - w * qz), 2 * (x * qz + w * y),
                      2 * (x * y + w * qz), 1 - 2 * (x * x + qz * qz), 2 * (y * qz - w * x),
                      2 * (x * qz - w * y), 2 * (y * qz + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    P = (J @ R) @ (Rq * torch.exp(ls)[:, None, :])
    S = P @ P.transpose(1, 2)
    a, b, c = S[:, 0, 0] + DILATION, S[:, 0, 1], S[:, 1, 1] + DILATION
    det = a * c - b * b
    conic = torch.stack([c / det, -b / det, a / det], 1)
    with torch.no_grad():
        lam = 0.5 * (a + c) + torch.sqrt(torch.clamp((0.5 * (a - c)) ** 2 + b * b, min=0.1))
        radius = torch.ceil(3 * torch.sqrt(lam))
    uv = torch.stack([cam.fx * xy[:, 0] + cam.cx, cam.fy * xy[:, 1] + cam.cy], 1)
    pos = -(R.T @ t)
    d = torch.nn.functional.normalize(mu - pos, dim=1)
    rgb = torch.relu((_sh_basis(deg, d)[:, :, None] * sh).sum(1) + 0.5)
    return uv, conic, torch.sigmoid(logit), rgb, radius


def _lists64(params32, cam, uv, radius):
    """Pairs (tile, Gaussian) of the 3-sigma squares by tile, then front to back: the depth key
    is the 32-bit depth ((R6 x + R7 y) + R8 z) + t2, each operation rounded, ties by index."""
    mu = params32[0]
    R = torch.tensor(cam.R, device=DEV)
    depth = (mu[:, 0] * R[2, 0] + mu[:, 1] * R[2, 1]) + mu[:, 2] * R[2, 2]
    depth = depth + float(cam.t[2])
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    r = radius[:, None]
    lo = torch.floor((uv - r) / 16).clamp(min=0)
    hi = torch.floor((uv + r) / 16) + 1
    x0, y0 = lo[:, 0].clamp(max=tx).long(), lo[:, 1].clamp(max=ty).long()
    x1, y1 = hi[:, 0].clamp(0, tx).long(), hi[:, 1].clamp(0, ty).long()
    cnt = ((x1 - x0) * (y1 - y0)).clamp(min=0)
    cnt = torch.where((depth > NEAR) & (x1 > x0) & (y1 > y0), cnt, torch.zeros_like(cnt))
    order = torch.sort(depth, stable=True).indices
    cnt_o = cnt[order]
    ids = torch.repeat_interleave(order, cnt_o)
    k = torch.arange(ids.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt_o, 0) - cnt_o, cnt_o)
    wd = (x1 - x0)[ids]
    tile = (y0[ids] + k // wd) * tx + x0[ids] + k % wd
    tile, at = torch.sort(tile, stable=True)
    ids = ids[at]
    counts = torch.bincount(tile, minlength=tx * ty)
    return ids, counts, torch.cumsum(counts, 0) - counts, tx


def _tile_batches(counts, budget):
    """Tiles with entries, grouped by list length so that a padded batch stays in the budget."""
    c = counts.cpu().numpy()
    todo = np.argsort(-c, kind="stable")
    todo = todo[c[todo] > 0]
    i = 0
    while i < len(todo):
        L = int(c[todo[i]])
        k = max(1, budget // (L * 256))
        yield todo[i:i + k], L
        i += k


class _Blend:
    """One batch of tiles in 64 bits: alphas [tiles, L, 256] of the staged lists."""

    def __init__(self, tiles, L, ids, counts, start, tx, sp):
        t = torch.from_numpy(tiles).to(DEV)
        pos = torch.arange(L, device=DEV)
        self.have = pos[None] < counts[t][:, None]
        self.g = ids[torch.where(self.have, start[t][:, None] + pos[None], torch.zeros_like(pos)[None])]
        px = torch.arange(256, device=DEV)
        self.x = (t % tx)[:, None] * 16 + px % 16
        self.y = torch.div(t, tx, rounding_mode="floor")[:, None] * 16 + px // 16
        uv, conic, op, rgb = sp
        m = uv[self.g]
        self.dx = (self.x[:, None] + 0.5) - m[..., 0:1]
        self.dy = (self.y[:, None] + 0.5) - m[..., 1:2]
        q = conic[self.g]
        self.q, self.rgb = q, rgb[self.g]
        sg = 0.5 * (q[..., 0:1] * self.dx ** 2 + q[..., 2:3] * self.dy ** 2) + q[..., 1:2] * self.dx * self.dy
        self.G = torch.exp(-sg)
        raw = op[self.g][..., None] * self.G
        self.clip = raw > ALPHA_MAX
        a = raw.clamp(max=ALPHA_MAX)
        self.use = (sg >= 0) & (a >= _f32(ALPHA_MIN)) & self.have[..., None]
        a = torch.where(self.use, a, torch.zeros_like(a))
        after = torch.cumprod(1 - a, 1)
        self.use &= after >= _f32(T_MIN)                   # the pixel stops before this entry
        self.a = torch.where(after >= _f32(T_MIN), a, torch.zeros_like(a))
        del a, raw, sg, after
        keep = torch.cumprod(1 - self.a, 1)
        self.T = torch.cat([torch.ones_like(keep[:, :1]), keep[:, :-1]], 1)
        self.Tf = keep[:, -1]                              # [tiles, 256]
        self.w = self.a * self.T
        self.C = torch.einsum("tlp,tlc->tpc", self.w, self.rgb)


def _render64(lists, sp, cam, budget=1 << 24):
    """A (premultiplied colour and 1 - T) [H, W, 4] of the block alone."""
    ids, counts, start, tx = lists
    A = torch.zeros(cam.height, cam.width, 4, dtype=torch.float64, device=DEV)
    for tiles, L in _tile_batches(counts, budget):
        b = _Blend(tiles, L, ids, counts, start, tx, sp)
        ok = (b.x < cam.width) & (b.y < cam.height)
        A[b.y[ok], b.x[ok]] = torch.cat([b.C, 1 - b.Tf[..., None]], -1)[ok]
    return A


def _render64_grad(lists, sp, cam, gA, budget=1 << 24):
    """Gradients of uv, conic, opacity and colour for dL/dA = gA [H, W, 4]."""
    ids, counts, start, tx = lists
    n = sp[0].shape[0]
    out = torch.zeros(n, 9, dtype=torch.float64, device=DEV)
    for tiles, L in _tile_batches(counts, budget):
        b = _Blend(tiles, L, ids, counts, start, tx, sp)
        ok = (b.x < cam.width) & (b.y < cam.height)
        gp = torch.zeros(*b.x.shape, 4, dtype=torch.float64, device=DEV)
        gp[ok] = gA[b.y[ok], b.x[ok]]
        gc = torch.einsum("tlc,tpc->tlp", b.rgb, gp[..., :3])            # G . colour
        inc = torch.cumsum(b.w * gc, 1)
        K = (gp[..., :3] * b.C).sum(-1) - gp[..., 3] * b.Tf
        da = b.T * gc - (K[:, None] - inc) / (1 - b.a)
        da = torch.where(b.use & ~b.clip, da, torch.zeros_like(da))
        ds = -da * b.a                                                    # d alpha / d sigma = -alpha
        q = b.q
        parts = [-(q[..., 0:1] * b.dx + q[..., 1:2] * b.dy) * ds, -(q[..., 2:3] * b.dy + q[..., 1:2] * b.dx) * ds,
                 0.5 * b.dx ** 2 * ds, b.dx * b.dy * ds, 0.5 * b.dy ** 2 * ds, da * b.G]
        g9 = torch.cat([torch.stack([p.sum(-1) for p in parts], -1),
                        torch.einsum("tlp,tpc->tlc", b.w, gp[..., :3])], -1)
        out.index_add_(0, b.g[b.have], g9[b.have])
    return out


def _loss64(x, y):
    """(1 - lam) L1 + lam (1 - SSIM), 11x11 Gaussian window of sigma 1.5, zero padding."""
    w = torch.exp(-(torch.arange(11, dtype=torch.float64, device=DEV) - 5) ** 2 / 4.5)
    w = (w / w.sum())

    def win(v):
        v = torch.nn.functional.conv2d(v, w.view(1, 1, 11, 1), padding=(5, 0))
        return torch.nn.functional.conv2d(v, w.view(1, 1, 1, 11), padding=(0, 5))

    a, b = x.permute(2, 0, 1)[:, None], y.permute(2, 0, 1)[:, None]
    ma, mb = win(a), win(b)
    va, vb, cab = win(a * a) - ma * ma, win(b * b) - mb * mb, win(a * b) - ma * mb
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    s = (2 * ma * mb + c1) * (2 * cab + c2) / ((ma * ma + mb * mb + c1) * (va + vb + c2))
    return (1 - LAM) * (x - y).abs().mean() + LAM * (1 - s.mean())


def _exact_step(case, seed):
    params32, cam = _block(case, seed)
    F, B, gt = _images(case, seed)
    params = [t.double().requires_grad_(True) for t in params32]
    uv, conic, op, rgb, radius = _project64(params, cam, case["sh"])
    sp = [v.detach() for v in (uv, conic, op, rgb)]
    lists = _lists64(params32, cam, sp[0], radius)
    A = _render64(lists, sp, cam).requires_grad_(True)
    zero = torch.zeros(case["h"], case["w"], 4, dtype=torch.float64, device=DEV)
    F, B = (zero if v is None else v.double() for v in (F, B))
    bg = torch.tensor([_f32(v) for v in (_bg(case) or (0.0, 0.0, 0.0))], dtype=torch.float64, device=DEV)
    full = F + (1 - F[..., 3:]) * (A + (1 - A[..., 3:]) * B)
    out = torch.cat([full[..., :3] + (1 - full[..., 3:]) * bg, full[..., 3:]], -1)
    loss = _loss64(out[..., :3], gt.double())
    gA = torch.autograd.grad(loss, A)[0]
    g9 = _render64_grad(lists, sp, cam, gA)
    grads = torch.autograd.grad([uv, conic, op, rgb], params, [g9[:, 0:2], g9[:, 2:5], g9[:, 5], g9[:, 6:9]])
    res = {"out": out.detach(), "loss": loss.detach().view(1), "grads": [g.contiguous() for g in grads]}
    if case["kind"] == "grad":
        return res
    m0, v0 = _moments(params32, seed)
    b1, b2, t = _f32(BETA1), _f32(BETA2), STEP0 + 1
    lr = [_f32(x) for x in _lr(case)]
    th, ms, vs = [], [], []
    for k, (p, g) in enumerate(zip(params, grads)):
        m = b1 * m0[k].double() + (1 - b1) * g
        v = b2 * v0[k].double() + (1 - b2) * g * g
        rate = torch.full_like(p, lr[k]).detach()
        if k == 4:
            rate[:, 1:] = lr[5]
        th.append(p.detach() - rate * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + _f32(EPS)))
        ms.append(m)
        vs.append(v)
    return {**res, "theta": th, "m": ms, "v": vs}


def _stored_tiles(lists, sp):
    """Whether a tile is stored: some Gaussian of its square comes within the listing margin of
    alpha_min on the box of the tile's pixel centres."""
    ids, counts, start, tx = lists
    tile = torch.repeat_interleave(torch.arange(counts.numel(), device=DEV), counts)
    uv, conic, op, _ = sp
    near = torch.zeros(counts.numel(), dtype=torch.bool, device=DEV)
    for k in range(0, ids.numel(), 1 << 22):
        g, t = ids[k:k + (1 << 22)], tile[k:k + (1 << 22)]
        X0 = (t % tx) * 16 + 0.5 - uv[g, 0]
        Y0 = torch.div(t, tx, rounding_mode="floor") * 16 + 0.5 - uv[g, 1]
        a, b, c = (0.5 * conic[g, 0], conic[g, 1], 0.5 * conic[g, 2])
        best = torch.full_like(X0, math.inf)
        for e in (0.0, 15.0):
            X, Y = X0 + e, Y0 + e
            dy = torch.minimum(torch.maximum(-b * X / (2 * c), Y0), Y0 + 15)
            best = torch.minimum(best, a * X * X + b * X * dy + c * dy * dy)
            dx = torch.minimum(torch.maximum(-b * Y / (2 * a), X0), X0 + 15)
            best = torch.minimum(best, a * dx * dx + b * dx * Y + c * Y * Y)
        inside = (X0 <= 0) & (X0 + 15 >= 0) & (Y0 <= 0) & (Y0 + 15 >= 0)
        best = torch.where(inside, torch.zeros_like(best), best) / math.log(2.0)
        thr = torch.log2(op[g] / _f32(ALPHA_MIN))
        ok = (op[g] >= _f32(ALPHA_MIN)) & (best <= (1.001 * thr + 0.01) * 1.001)
        near[t[ok]] = True
    return near


def _exact_refresh(case, seed):
    params32, cam = _block(case, seed)
    uv, conic, op, rgb, radius = _project64([t.double() for t in params32], cam, case["sh"])
    sp = [uv, conic, op, rgb]
    lists = _lists64(params32, cam, uv, radius)
    A = _render64(lists, sp, cam)
    if case["kind"] == "refresh_dense":
        return A
    tx, ty = (case["w"] + 15) // 16, (case["h"] + 15) // 16
    pad = torch.zeros(ty * 16, tx * 16, 4, dtype=torch.float64, device=DEV)
    pad[:case["h"], :case["w"]] = A
    blocks = pad.view(ty, 16, tx, 16, 4).permute(0, 2, 1, 3, 4).reshape(tx * ty, 16, 16, 4)
    stored = blocks[_stored_tiles(lists, sp)]
    packed = torch.zeros_like(blocks)
    packed[:stored.shape[0]] = stored
    return {"map": None, "packed": packed, "count": None}


def _decode(tile_map, data, case):
    tx, ty = (case["w"] + 15) // 16, (case["h"] + 15) // 16
    t = torch.where((tile_map >= 0)[:, None, None, None], data[tile_map.clamp(min=0).long()].double(),
                    torch.zeros((), dtype=torch.float64, device=DEV))
    return t.view(ty, tx, 16, 16, 4).permute(0, 2, 1, 3, 4).reshape(ty * 16, tx * 16, 4)[:case["h"], :case["w"]]


def _fold64(layers, case):
    acc = torch.zeros(case["h"], case["w"], 4, dtype=torch.float64, device=DEV)
    for x in layers:
        acc = acc + (1 - acc[..., 3:]) * x.double()
    return acc


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "grad", "refresh_packed", "refresh_dense"):
        covered, _ = _splat_work(case)
        # pairs of the lists, roughly: beyond these the padded batches take over 20 seconds
        f = 0.5 * case["w"] / math.tan(math.radians(30.0))
        radius = 30.0 if case["grid"] == "mixture" else 1.5 * _half_diag(_dims(case))
        if case["n"] * (6.0 * f * 0.05 * SIDE / radius / 16 + 1.5) ** 2 > 6e7:
            return None
        return _exact_step(case, seed) if kind in ("step", "grad") else _exact_refresh(case, seed)
    order, split = _order(case, seed)
    if kind in ("composite", "eval"):
        dt = torch.float32 if case.get("dtype") == "f32" else torch.float16
        layers = _dense_layers(case, seed, dt)
        if kind == "composite":
            return [_fold64([layers[k] for k in order[:split]], case),
                    _fold64([layers[k] for k in order[split + 1:]], case)]
        full = _fold64([layers[k] for k in order], case)
        return [full, _loss64(full[..., :3], _images({**case, "fb": "none"}, seed)[2].double()).view(1)]
    maps, data = _packed_layers(case, seed)
    dec = lambda k: _decode(maps[k], data[k], case)
    if kind == "composite_packed":
        return [_fold64(map(dec, order[:split]), case), _fold64(map(dec, order[split + 1:]), case)]
    if kind == "fold_packed":
        acc = _fold64(map(dec, order), case)
        return [acc, acc]
    T = torch.ones(case["h"], case["w"], dtype=torch.float64, device=DEV)
    vis, cov = (torch.zeros(case["layers"], dtype=torch.float64, device=DEV) for _ in range(2))
    for k in order:
        a = dec(k)[..., 3]
        vis[k], cov[k] = (a * T).mean(), a.mean()
        T = T * (1 - a)
    return [vis, cov]
