"""The work whose speed is measured: the library's imaging pipelines, realized
through the Python binding as a program that filters images calls them.

A program builds a pipeline once, gives it the stored schedule of its kind that
is nearest in size (``tuner``), reserves what it needs for the image size, and
then realizes it on device images, as CUDA graph replays, on torch's current
stream.  A pass is one image.
"""

import math

import numpy as np
import torch

from paper_2012_07145_gb300 import hp, pipelines, tuner

STORAGE = {"f32": hp.HP_F32, "f16": hp.HP_F16, "bf16": hp.HP_BF16, "u8": hp.HP_U8, "u16": hp.HP_U16}
# 16-bit integers are held as int16 bits, as everywhere in this repository
TORCH = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "u8": torch.uint8, "u16": torch.int16}
IN_CHANNELS = {"chain": 1, "harris": 3, "unsharp": 3, "histeq": 1, "laplacian": 3, "maxfilter": 3, "interpolate": 4,
               "bilateral": 1}
OUT_CHANNELS = {**IN_CHANNELS, "harris": 1, "interpolate": 3}
# the largest image of each application, in pixels: the benchmark's sizes
LARGEST = {"chain": 2560 * 1536, "harris": 4096 * 3072, "unsharp": 4096 * 3072, "histeq": 4096 * 3072,
           "laplacian": 2560 * 1536, "maxfilter": 2560 * 1536, "interpolate": 2560 * 1536, "bilateral": 2560 * 1536}
SMALLEST = 256 * 256


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # a short blur of a thumbnail: one small launch, where latency counts
        dict(name="chain4_512x512_f32", app="chain", w=512, h=512, dtype="f32", stages=4, pattern="binomial"),
        # the headline: the 32-stage stencil chain at the benchmark's size
        dict(name="chain32_2560x1536_f32", app="chain", w=2560, h=1536, dtype="f32", stages=32, pattern="alternate"),
        # the same chain kept in 16 bits, on a full-HD frame whose width and height are odd
        dict(name="chain32_1919x1079_bf16", app="chain", w=1919, h=1079, dtype="bf16", stages=32,
             pattern="alternate"),
        # corner response of a camera frame for tracking: one request of the serving mix
        dict(name="harris_640x480_f32", app="harris", w=640, h=480, dtype="f32"),
        # corner response of a photograph
        dict(name="harris_2560x1536_f32", app="harris", w=2560, h=1536, dtype="f32"),
        # sharpening the largest photograph of the serving mix
        dict(name="unsharp_4096x3072_f32", app="unsharp", w=4096, h=3072, dtype="f32"),
        # sharpening a web-size picture, ragged rows
        dict(name="unsharp_1023x767_f32", app="unsharp", w=1023, h=767, dtype="f32"),
        # contrast equalization of a large 8-bit photograph
        dict(name="histeq_4096x3072_u8", app="histeq", w=4096, h=3072, dtype="u8"),
        # tone mapping: the benchmark's local Laplacian
        dict(name="laplacian_2560x1536_u16", app="laplacian", w=2560, h=1536, dtype="u16", levels=8, alpha=1.0),
        # 9 x 9 dilation per channel
        dict(name="maxfilter_2560x1536_f32", app="maxfilter", w=2560, h=1536, dtype="f32", radius=4),
        # filling the uncovered pixels of a sparsely sampled image, odd at every level
        dict(name="interpolate_2559x1535_f32", app="interpolate", w=2559, h=1535, dtype="f32", levels=10),
        # edge-preserving smoothing of a gray photograph
        dict(name="bilateral_2560x1536_f32", app="bilateral", w=2560, h=1536, dtype="f32"),
    ]


def draw(rng):
    app = rng.choice(sorted(IN_CHANNELS))
    # pixels and aspect over their logarithms; any width and height, odd ones among them
    pixels = math.exp(rng.uniform(math.log(SMALLEST), math.log(LARGEST[app])))
    aspect = math.exp(rng.uniform(math.log(0.6), math.log(2.0)))
    w = max(128, round(math.sqrt(pixels * aspect)))
    h = max(128, min(round(pixels / w), LARGEST[app] // w))
    case = dict(app=app, w=w, h=h, dtype="f32")
    if app == "chain":
        case.update(stages=rng.choice([4, 8, 16, 32]), pattern=rng.choice(["alternate", "binomial"]),
                    dtype=rng.choice(["f32", "f32", "f16", "bf16"]))
    elif app == "harris":
        case.update(dtype=rng.choice(["f32", "f32", "bf16"]))
    elif app == "histeq":
        case.update(dtype="u8")
    elif app == "laplacian":
        case.update(dtype="u16", levels=rng.choice([6, 7, 8]), alpha=rng.choice([0.25, 0.5, 1.0]))
    elif app == "maxfilter":
        case.update(radius=rng.choice([1, 2, 3, 4]), dtype=rng.choice(["f32", "f32", "bf16"]))
    elif app == "interpolate":
        case.update(levels=rng.choice([6, 8, 10]))
    return case


# ------------------------------------------------------------------ inputs --
def image(case, seed):
    """The case's input image [C][H][W] on the GPU, in its storage type."""
    app, w, h = case["app"], case["w"], case["h"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = IN_CHANNELS[app]

    def uniform(n):
        return torch.rand((n, h, w), generator=g, device="cuda")

    def ramp_noise(base, sigma):
        return (base + sigma * torch.randn(base.shape, generator=g, device="cuda")).clamp_(0.0, 1.0)

    xs = (torch.arange(w, device="cuda") / max(w - 1, 1)).expand(h, w)
    ys = (torch.arange(h, device="cuda") / max(h - 1, 1))[:, None].expand(h, w)
    if app == "histeq":        # low contrast: N(100, 20)
        return (100.0 + 20.0 * torch.randn((1, h, w), generator=g, device="cuda")).round_().clamp_(0, 255).to(torch.uint8)
    if app == "laplacian":     # smooth gradients and camera noise, 16 bits a channel
        v = ramp_noise(torch.stack([xs, ys, (xs + ys) / 2]), 0.02)
        return (v * 65535.0).round_().to(torch.int32).to(torch.int16)
    if app == "bilateral":     # a gradient with noise to remove
        return ramp_noise(((xs + ys) / 2)[None], 0.05)
    if app == "interpolate":   # colours known at a quarter of the pixels
        return torch.cat([uniform(3), (uniform(1) < 0.25).float()])
    return uniform(c).to(TORCH[case["dtype"]])


# ------------------------------------------------------------------ passes --
def nearest_entry(pipeline, w, h, dtype):
    """The stored schedule of this pipeline and type nearest in pixels, or None."""
    best = None
    for k, entry in tuner.load_db().items():
        name, ew, eh, ed = tuner.parse_key(k)
        if name == pipeline and ed == dtype:
            off = abs(math.log((ew * eh) / (w * h)))
            if best is None or off < best[0]:
                best = (off, entry)
    return best[1] if best else None


def build(case):
    """The case's pipeline with its schedule."""
    app, w, h, dtype = case["app"], case["w"], case["h"], case["dtype"]
    st = STORAGE[dtype]
    if app == "chain":
        p = pipelines.stencil_chain(case["stages"], case["pattern"], storage=st)
        stored = "stencil_chain_4_binomial" if case["stages"] == 4 and dtype == "f32" else "stencil_chain_32_alternate"
        tuner.apply_entry(p, None, stored, nearest_entry(stored, w, h, dtype))
    elif app == "laplacian":
        p, ids = pipelines.local_laplacian(levels=case["levels"], k_levels=8, alpha=case["alpha"])
        tuner.apply_entry(p, ids, "local_laplacian_J8_K8", nearest_entry("local_laplacian_J8_K8", w, h, dtype))
    elif app == "interpolate":
        p, ids = pipelines.interpolate(case["levels"])
        pipelines.interpolate_fused_schedule(p, ids)
    elif app == "bilateral":
        p = pipelines.bilateral_grid(8, 0.1)
        pipelines.bilateral_grid_fused_schedule(p)
    elif app == "maxfilter":
        p = pipelines.max_filter(case["radius"], io_storage=st)
        p.schedule([0, 0])
    else:
        p = {"harris": lambda: pipelines.harris(io_storage=st, inner_storage=st), "unsharp": pipelines.unsharp,
             "histeq": pipelines.histeq}[app]()
        tuner.apply_entry(p, None, app, nearest_entry(app, w, h, dtype))
    return p


def prepare(case, seed):
    w, h, dtype = case["w"], case["h"], case["dtype"]
    p = build(case)
    p.use_cuda_graph(True)
    stream = torch.cuda.current_stream().cuda_stream
    p.prepare([(w, h)], stream)
    x = hp.padded_copy(image(case, seed))
    y = hp.padded_empty(OUT_CHANNELS[case["app"]], h, w, TORCH[dtype])
    return dict(p=p, inputs=[hp.buffer_from_tensor(x, STORAGE[dtype])], output=hp.buffer_from_tensor(y, STORAGE[dtype]),
                y=y)


def run(state):
    state["p"].realize(state["inputs"], state["output"], torch.cuda.current_stream().cuda_stream)
    return state["y"]


def work(case):
    """Bytes: the image read once and the result written once.  Operations, per
    pixel: a separable 5 x 5 stage 14 (binomial) or 10 (box); Harris 68; unsharp
    14 + 3 per channel; the local Laplacian 125 for the remapped first level of
    its pyramid, a third more for the coarser ones and 100 for interpolation
    and collapse; a window maximum 2 log2(window) per channel; the interpolate
    pyramid 4 channels of 20 and the composites; the bilateral slice 50."""
    app, px = case["app"], case["w"] * case["h"]
    size = {"f32": 4, "f16": 2, "bf16": 2, "u8": 1, "u16": 2}[case["dtype"]]
    if app == "chain":
        n = case["stages"]
        ops = 14 * n if case["pattern"] == "binomial" else 12 * n
    else:
        ops = {"harris": 68, "unsharp": 51, "histeq": 2, "laplacian": 266, "interpolate": 110, "bilateral": 55,
               "maxfilter": 3 * 2 * math.ceil(math.log2(2 * case.get("radius", 1) + 1))}[app]
    return dict(bytes=px * size * (IN_CHANNELS[app] + OUT_CHANNELS[app]), flops=px * ops)


# ----------------------------------------------------- the results in 64 bits --
def clamped(x, dim, offset, stride=1, n=None):
    """x at the indices stride * i + offset, clamped to its extent, along dim."""
    n = x.shape[dim] if n is None else n
    i = (torch.arange(n, device=x.device) * stride + offset).clamp_(0, x.shape[dim] - 1)
    return x.index_select(dim, i)


def separable(x, wx, wy):
    for dim, taps in ((-1, wx), (-2, wy)):
        r = len(taps) // 2
        x = sum(t * clamped(x, dim, k - r) for k, t in enumerate(taps) if t)
    return x


BINOMIAL = [1 / 16, 4 / 16, 6 / 16, 4 / 16, 1 / 16]


def down(x):
    for dim in (-1, -2):
        n = (x.shape[dim] + 1) // 2
        x = sum(t * clamped(x, dim, k - 2, 2, n) for k, t in enumerate(BINOMIAL))
    return x


def up(x, shape):
    for dim, n in ((-1, shape[-1]), (-2, shape[-2])):
        m = torch.arange(n, device=x.device) // 2
        at = lambda k: x.index_select(dim, (m + k).clamp_(0, x.shape[dim] - 1))  # noqa: E731
        odd = (torch.arange(n, device=x.device) % 2 == 1)
        odd = odd if dim == -1 else odd[:, None]
        x = torch.where(odd, (at(0) + at(1)) / 2, (at(-1) + 6 * at(0) + at(1)) / 8)
    return x


def gray(x):
    return 0.299 * x[0] + 0.587 * x[1] + 0.114 * x[2]


def exact_laplacian(x, levels, alpha, sigma=0.1, K=8):
    x = (x.to(torch.int32) & 0xFFFF).double() / 65535
    g = gray(x)
    d = g[None] - torch.arange(K, device=x.device, dtype=torch.float64)[:, None, None] / (K - 1)
    m = torch.where(d.abs() <= sigma, sigma * (d.abs() / sigma) ** alpha, d.abs())
    G = [torch.cat([g[None] - d + torch.sign(d) * m, g[None]])]
    for _ in range(levels - 1):
        G.append(down(G[-1]))
    r = G[-1][K]
    for fine, coarse in zip(G[-2::-1], G[:0:-1]):
        lap = fine[:K] - up(coarse[:K], fine.shape)
        t = fine[K] * (K - 1)
        k0 = t.floor().long().clamp_(0, K - 2)
        f = t - k0
        lo, hi = (lap.gather(0, (k0 + k)[None])[0] for k in (0, 1))
        r = (1 - f) * lo + f * hi + up(r, fine.shape)
    out = torch.where(g > 0, x * (r / torch.where(g > 0, g, 1.0)), r)
    return (out * 65535).round().clamp_(0, 65535).to(torch.int32).to(torch.int16)


def exact_interpolate(x, levels):
    x = x.double()
    D = [torch.cat([x[:3] * x[3:], x[3:]])]
    for _ in range(levels - 1):
        D.append(down(D[-1]))
    r = D[-1]
    for fine in D[-2::-1]:
        r = fine + (1 - fine[3:]) * up(r, fine.shape)
    return torch.where(r[3:] > 0, r[:3] / torch.where(r[3:] > 0, r[3:], 1.0), 0.0)


def exact_bilateral(x, s=8, r=0.1):
    r = float(np.float32(r))
    gz = int(math.floor(1 / r + 0.5)) + 1
    v = x[0].double().clamp(0, 1)
    h, w = v.shape
    gh, gw = -(-h // s) + 1, -(-w // s) + 1
    # the range level is decided in 32 bits, part of the filter's definition
    inv = np.float64(np.float32(1 / r))
    rows = (torch.arange(gh * s, device=v.device) - s // 2).clamp_(0, h - 1)
    cols = (torch.arange(gw * s, device=v.device) - s // 2).clamp_(0, w - 1)
    c = v[rows][:, cols]
    z = (c * inv + 0.5).float().floor().long().clamp_(0, gz - 1)
    cell = (torch.arange(gh * s, device=v.device) // s)[:, None] * gw + (torch.arange(gw * s, device=v.device) // s)
    grid = torch.zeros((2, gh * gw * gz), dtype=torch.float64, device=v.device)
    at = (cell * gz + z).reshape(-1)
    grid[0].scatter_add_(0, at, c.reshape(-1))
    grid[1].scatter_add_(0, at, torch.ones_like(c).reshape(-1))
    grid = grid.reshape(2, gh, gw, gz)
    for dim in (3, 2, 1):
        grid = sum(t * clamped(grid, dim, k - 2) for k, t in enumerate(BINOMIAL))
    zf = v / r
    xf = (torch.arange(w, device=v.device, dtype=torch.float64) / s).expand(h, w)
    yf = (torch.arange(h, device=v.device, dtype=torch.float64) / s)[:, None].expand(h, w)
    acc = 0
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                part = 1.0
                at = []
                for f, d, n in ((yf, dy, gh), (xf, dx, gw), (zf, dz, gz)):
                    f0 = f.floor()
                    part = part * ((f - f0) if d else (1 - (f - f0)))
                    at.append((f0.long() + d).clamp_(0, n - 1))
                acc = acc + part * grid[:, at[0], at[1], at[2]]
    return torch.where(acc[1] > 0, acc[0] / torch.where(acc[1] > 0, acc[1], 1.0), v)[None]


def exact(case, seed):
    app = case["app"]
    x = image(case, seed)
    if app == "laplacian":
        return exact_laplacian(x, case["levels"], case["alpha"])
    if app == "interpolate":
        return exact_interpolate(x, case["levels"])
    if app == "bilateral":
        return exact_bilateral(x)
    if app == "histeq":
        n = torch.bincount(x.reshape(-1).long(), minlength=256).cpu().tolist()
        cdf = [sum(n[: v + 1]) for v in range(256)]
        first = next(c for c in cdf if c)
        total = cdf[-1]
        if total == first:
            return x
        lut = [max(0, (2 * 255 * (c - first) + (total - first)) // (2 * (total - first))) for c in cdf]
        return torch.tensor(lut, dtype=torch.uint8, device=x.device)[x.long()]
    x = x.double()
    if app == "chain":
        for k in range(case["stages"]):
            taps = [0.2] * 5 if case["pattern"] == "alternate" and k % 2 else BINOMIAL
            x = separable(x, taps, taps)
        return x
    if app == "harris":
        g = gray(x)
        ix, iy = separable(g, [-1, 0, 1], [1, 2, 1]), separable(g, [1, 2, 1], [-1, 0, 1])
        sxx, syy, sxy = (separable(v, [1, 1, 1], [1, 1, 1]) for v in (ix * ix, iy * iy, ix * iy))
        return (sxx * syy - sxy * sxy - 0.04 * (sxx + syy) ** 2)[None]
    if app == "unsharp":
        return x + 1.5 * (x - separable(x, BINOMIAL, BINOMIAL))
    r = case["radius"]   # maxfilter
    for dim in (-1, -2):
        y = x
        for k in range(-r, r + 1):
            y = torch.maximum(y, clamped(x, dim, k))
        x = y
    return x
