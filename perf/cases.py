"""The calls whose time is tracked: GFC solves, their adjoint and edits as user programs make them.

Every case goes through the public Python entry points (``gfc.Plan``,
``gfc.RaggedPlan``, ``gfc.gfc_layer``). Inputs are image-like: smooth images
with texture, their forward-difference gradients, and the edits the method is
used for (a region whose gradient is removed, rectangles of added gradient, a
patch whose gradient comes from another image), or box-blurred Gaussian feature
maps for the layer. ``exact`` restates the solve with torch's FP64 FFTs.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1902_00176_gb300 import gfc

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
PAD = 4


def listed():
    return [
        # one small image with a region's gradient removed: an interactive edit, bound by latency
        {"name": "removal_64x96", "op": "solve", "edit": "remove", "batch": 1, "C": 1, "H": 64, "W": 96,
         "dtype": "f32"},
        # one colour photo after a gradient-domain edit, the size of the paper's timing
        {"name": "photo_rgb_801x1200", "op": "solve", "edit": "perturb", "batch": 1, "C": 3, "H": 801, "W": 1200,
         "dtype": "f32"},
        # the paper's batch of 100 Laplacian solves at 801x1200
        {"name": "batch100_801x1200", "op": "solve", "edit": "perturb", "batch": 100, "C": 1, "H": 801, "W": 1200,
         "dtype": "f32"},
        # Poisson blending of a batch of colour images kept in 16 bits
        {"name": "blend_f16_1024x1536", "op": "solve", "edit": "blend", "batch": 16, "C": 3, "H": 1024, "W": 1536,
         "dtype": "f16"},
        # cropped photos: odd sizes, rows that are not whole 16-byte vectors
        {"name": "crops_rgb_613x927", "op": "solve", "edit": "perturb", "batch": 8, "C": 3, "H": 613, "W": 927,
         "dtype": "f32"},
        # the Laplacian itself as the input (the form of the paper's Algorithm B)
        {"name": "laplacian_512x512", "op": "laplacian", "edit": "perturb", "batch": 16, "C": 3, "H": 512, "W": 512,
         "dtype": "f32"},
        # texture flattening: gradient threshold, solve and colour correction in one call
        {"name": "flatten_rgb_720x1080", "op": "flatten", "edit": "none", "batch": 8, "C": 3, "H": 720, "W": 1080,
         "dtype": "f32"},
        # the merging layer on the feature maps of a batch, forward and backward
        {"name": "layer_bf16_256x256", "op": "layer", "edit": "features", "batch": 32, "C": 64, "H": 256, "W": 256,
         "dtype": "bf16"},
        # the same layer deeper in a network: small maps, many channels
        {"name": "layer_bf16_64x64", "op": "layer", "edit": "features", "batch": 32, "C": 128, "H": 64, "W": 64,
         "dtype": "bf16"},
        # training through the solve on colour images of the width of a data set's photos, odd sizes
        {"name": "train_rgb_375x499", "op": "layer", "edit": "perturb", "batch": 16, "C": 3, "H": 375, "W": 499,
         "dtype": "f32"},
        # photos of all sizes, solved as one ragged batch
        {"name": "ragged64_128_2000", "op": "ragged", "edit": "perturb", "items": 64, "lo": 128, "hi": 2000,
         "sizes": 7, "dtype": "f32"},
        # one large colour photo
        {"name": "photo_rgb_2160x3840", "op": "solve", "edit": "remove", "batch": 1, "C": 3, "H": 2160, "W": 3840,
         "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "laplacian", "flatten", "layer", "layer", "ragged"])
    if op == "ragged":
        lo = _log_int(rng, 48, 256)
        return {"op": op, "edit": "perturb", "items": _log_int(rng, 8, 64), "lo": lo,
                "hi": _log_int(rng, 4 * lo, 2000), "sizes": rng.randrange(1 << 20), "dtype": "f32"}
    if op == "layer":  # feature maps in 16 bits, or colour images in 32
        maps = rng.random() < 0.6
        H = _log_int(rng, 28, 320) if maps else _log_int(rng, 96, 1024)
        W = max(24, int(H * rng.uniform(0.75, 1.5)))
        C = rng.choice([16, 32, 64, 96, 128]) if maps else rng.choice([1, 3])
        most = 6.0e7 if maps else 2.0e7
        return {"op": op, "edit": "features" if maps else "perturb",
                "batch": _log_int(rng, 1, max(1, min(64, int(most / (C * H * W))))), "C": C, "H": H, "W": W,
                "dtype": "bf16" if maps and rng.random() < 0.7 else ("f16" if maps else "f32")}
    H = _log_int(rng, 64, 2000)  # images: from thumbnails to large photos, portrait and landscape
    W = max(64, min(3840, int(H * rng.uniform(0.67, 1.78))))
    C = rng.choice([1, 3, 3])
    return {"op": op, "edit": "none" if op == "flatten" else rng.choice(["remove", "perturb", "blend"]),
            "batch": _log_int(rng, 1, max(1, min(128, int(4.0e7 / (C * H * W))))), "C": C, "H": H, "W": W,
            "dtype": "f32" if op != "solve" else rng.choice(["f32", "f32", "f16", "bf16"])}


# ---- inputs ----
def _images(gen, B, C, H, W):
    """Smooth random images in [0, 1] with a little texture."""
    low = torch.rand((B, C, max(4, H // 24 + 3), max(4, W // 24 + 3)), generator=gen, device="cuda")
    img = F.interpolate(low, size=(H, W), mode="bicubic", align_corners=True).clamp_(0.0, 1.0).mul_(0.95)
    return img.add_(torch.rand((B, C, H, W), generator=gen, device="cuda"), alpha=0.05)


def _gradient(img):
    """Forward differences, replicate border."""
    gx, gy = torch.zeros_like(img), torch.zeros_like(img)
    torch.sub(img[..., :, 1:], img[..., :, :-1], out=gx[..., :, :-1])
    torch.sub(img[..., 1:, :], img[..., :-1, :], out=gy[..., :-1, :])
    return gx, gy


def _edited(gen, host, edit, B, C, H, W):
    """(image, gx, gy) of a batch of images after `edit`, FP32."""
    img = _images(gen, B, C, H, W)
    gx, gy = _gradient(img)
    if edit == "remove":  # no gradient inside a quarter-size rectangle
        h, w = max(1, H // 4), max(1, W // 4)
        i, j = host.integers(0, H - h + 1), host.integers(0, W - w + 1)
        gx[..., i:i + h, j:j + w] = 0.0
        gy[..., i:i + h, j:j + w] = 0.0
    elif edit == "perturb":  # five rectangles of added gradient per component
        for g in (gx, gy):
            for _ in range(5):
                h, w = host.integers(max(1, H // 16), max(2, H // 4)), host.integers(max(1, W // 16), max(2, W // 4))
                i, j = host.integers(0, H - h + 1), host.integers(0, W - w + 1)
                g[..., i:i + h, j:j + w] += torch.rand((B, C, 1, 1), generator=gen, device="cuda") * 0.4 - 0.2
    elif edit == "blend":  # the gradient of another image inside an ellipse
        sx, sy = _gradient(_images(gen, B, C, H, W))
        ci, cj = H * host.uniform(0.35, 0.65), W * host.uniform(0.35, 0.65)
        ri, rj = H * host.uniform(0.1, 0.3), W * host.uniform(0.1, 0.3)
        i = (torch.arange(H, device="cuda") - ci) / ri
        j = (torch.arange(W, device="cuda") - cj) / rj
        mask = (i.square()[:, None] + j.square()[None, :]) <= 1.0
        gx, gy = torch.where(mask, sx, gx), torch.where(mask, sy, gy)
    return img, gx, gy


def _features(gen, B, C, H, W):
    x = torch.randn((B * C, 1, H, W), generator=gen, device="cuda")
    box = torch.full((1, 1, 5, 1), 0.2, device="cuda")
    x = F.conv2d(F.conv2d(x, box, padding=(2, 0)), box.view(1, 1, 1, 5), padding=(0, 2))
    return x.view(B, C, H, W)


def _ragged_items(case):
    r = np.random.default_rng(case["sizes"])
    return [(int(r.choice([1, 3])), int(r.integers(case["lo"], case["hi"] + 1)),
             int(r.integers(case["lo"], case["hi"] + 1))) for _ in range(case["items"])]


def _inputs(case, seed):
    """The case's input tensors by name, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 7919 + 17)
    host = np.random.default_rng(seed * 7919 + 17)
    dt = DTYPES[case["dtype"]]
    if case["op"] == "ragged":
        pairs = [_edited(gen, host, case["edit"], 1, C, H, W)[1:] for C, H, W in _ragged_items(case)]
        return {"gx": [p[0][0] for p in pairs], "gy": [p[1][0] for p in pairs]}
    B, C, H, W = case["batch"], case["C"], case["H"], case["W"]
    if case["edit"] == "features":
        s = {k: _features(gen, B, C, H, W).to(dt) for k in ("gx", "gy")}
    else:
        img, gx, gy = _edited(gen, host, case["edit"], B, C, H, W)
        if case["op"] == "laplacian":  # the divergence inside the image (backward differences)
            lap = gx + gy
            lap[..., :, 1:] -= gx[..., :, :-1]
            lap[..., 1:, :] -= gy[..., :-1, :]
            return {"lap": lap.to(dt)}
        s = {"gx": gx.to(dt), "gy": gy.to(dt)}
        if case["op"] == "flatten":  # the original image's statistics, which the result is rescaled to
            s["mean"] = img.mean(dim=(2, 3))
            s["std"] = img.std(dim=(2, 3), unbiased=False)
    if case["op"] == "layer":
        s["up"] = torch.randn((B, C, H, W), generator=gen, device="cuda").to(dt)
    return s


def prepare(case, seed):
    s = dict(_inputs(case, seed), op=case["op"])
    if case["op"] == "ragged":
        s["plan"] = gfc.RaggedPlan(_ragged_items(case), DTYPES[case["dtype"]])
        s["gx"], s["gy"] = s["plan"].pack(s["gx"]), s["plan"].pack(s["gy"])
    elif case["op"] == "layer":
        s["gx"].requires_grad_()
        s["gy"].requires_grad_()
    else:  # a program keeps one plan for all its images of a size
        s["plan"] = gfc.get_plan(case["H"], case["W"], case["C"], case["batch"], DTYPES[case["dtype"]],
                                 torch.device("cuda", torch.cuda.current_device()))
    return s


def run(s):
    if s["op"] == "layer":
        out = gfc.gfc_layer(s["gx"], s["gy"])
        ggx, ggy = torch.autograd.grad(out, (s["gx"], s["gy"]), s["up"])
        return {"out": out, "grad_gx": ggx, "grad_gy": ggy}
    if s["op"] == "laplacian":
        return s["plan"].solve_from_laplacian(s["lap"])
    if s["op"] == "flatten":
        return s["plan"].solve_corrected(s["gx"], s["gy"], s["mean"], s["std"], edit="threshold", frac=0.1)
    return s["plan"].solve_from_gradient(s["gx"], s["gy"])


# ---- what a pass cannot do without ----
def work(case):
    """Bytes: each input read once, each output written once. Operations: real transforms along
    one direction, forward and inverse, and some 20 operations a pixel for the rest."""
    if case["op"] == "ragged":
        sizes = [(C, H, W) for C, H, W in _ragged_items(case)]
    else:
        sizes = [(case["batch"] * case["C"], case["H"], case["W"])]
    n = sum(f * H * W for f, H, W in sizes)
    flops = sum(f * H * W * (5.0 * math.log2(W + 2 * PAD) + 20.0) for f, H, W in sizes)
    tensors, solves = {"laplacian": (2, 1), "layer": (6, 2)}.get(case["op"], (3, 1))
    return {"bytes": float(tensors * n * DTYPES[case["dtype"]].itemsize), "flops": float(flops * solves)}


# ---- the same in 64 bits ----
_ROW_LENGTHS = (108, 140, 160, 180, 200, 224, 252, 270, 294, 320, 360, 400, 448, 500, 560, 630, 700, 784, 882, 980,
                1080, 1120, 1200, 1250, 1372, 1400, 1536, 1568, 1750, 1960, 2058)


def _smooth_even(n):
    n += n & 1
    while True:
        m = n
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1:
            return n
        n += 2


def _torus(H, W):
    """The padded size (M, N) of an H x W image: even 7-smooth, rows from a list of lengths in its range."""
    n = W + 2 * PAD
    N = min(r for r in _ROW_LENGTHS if r >= n) if 136 < n <= _ROW_LENGTHS[-1] else _smooth_even(n)
    return _smooth_even(H + 2 * PAD), N


def _convolve(z):
    """Cyclic convolution of FP64 fields z [..., M, N] with the Green's function of the 5-point Laplacian."""
    M, N = z.shape[-2:]
    k = torch.sin(torch.arange(M, dtype=torch.float64, device=z.device) * (math.pi / M)).square_()
    l = torch.sin(torch.arange(N // 2 + 1, dtype=torch.float64, device=z.device) * (math.pi / N)).square_()
    lam = -4.0 * (k[:, None] + l[None, :])
    lam[0, 0] = 1.0
    S = torch.fft.rfft2(z).div_(lam)
    S[..., 0, 0] = 0.0
    return torch.fft.irfft2(S, s=(M, N))


def _solve64(lap, H, W):
    """Solve and crop; lap [f, M, N] is the right-hand side on the torus."""
    u = _convolve(lap)
    return u[..., PAD:PAD + H, PAD:PAD + W] - u[..., :1, :1]


def _divergence64(gx, gy, M, N):
    f, H, W = gx.shape
    z = torch.zeros((f, M, N), dtype=torch.float64, device=gx.device)
    z[:, PAD:PAD + H, PAD:PAD + W] += gx
    z[:, PAD:PAD + H, PAD + 1:PAD + W + 1] -= gx
    z[:, PAD:PAD + H, PAD:PAD + W] += gy
    z[:, PAD + 1:PAD + H + 1, PAD:PAD + W] -= gy
    return z


def _by_fields(fn, *tensors):
    """fn over [f, H, W] pieces of [B, C, H, W] tensors, some fields at a time."""
    B, C, H, W = tensors[0].shape
    step = max(1, int(1.0e8 / (H * W)))
    flat = [t.reshape(B * C, H, W) for t in tensors]
    parts = [fn(*(t[i:i + step].double() for t in flat)) for i in range(0, B * C, step)]
    join = lambda p: torch.cat(p).view(B, C, H, W)  # noqa: E731
    return tuple(join(p) for p in zip(*parts)) if isinstance(parts[0], tuple) else join(parts)


def exact(case, seed):
    s = _inputs(case, seed)
    if case["op"] == "ragged":
        flat, off = [], 0
        for (C, H, W), gx, gy in zip(_ragged_items(case), s["gx"], s["gy"]):
            M, N = _torus(H, W)
            u = _solve64(_divergence64(gx.double(), gy.double(), M, N), H, W).reshape(-1)
            flat.append(F.pad(u, (0, -u.numel() % 8)))  # items start at multiples of 8 elements
        return torch.cat(flat)
    H, W = case["H"], case["W"]
    M, N = _torus(H, W)
    if case["op"] == "laplacian":
        return _by_fields(lambda lap: _solve64(F.pad(lap, (PAD, N - W - PAD, PAD, M - H - PAD)), H, W), s["lap"])
    if case["op"] == "flatten":  # |E| below a tenth of the field's largest is dropped, decided in FP32
        m2 = s["gx"] * s["gx"] + s["gy"] * s["gy"]
        t = m2.amax(dim=(2, 3), keepdim=True).sqrt() * torch.tensor(0.1, dtype=torch.float32, device="cuda")
        drop = m2 < t * t
        s["gx"][drop] = 0.0
        s["gy"][drop] = 0.0
    out = _by_fields(lambda gx, gy: _solve64(_divergence64(gx, gy, M, N), H, W), s["gx"], s["gy"])
    if case["op"] == "flatten":
        mean, std = out.mean(dim=(2, 3), keepdim=True), out.std(dim=(2, 3), unbiased=False, keepdim=True)
        gain = s["std"].double()[..., None, None] / std
        return (out - mean) * gain + s["mean"].double()[..., None, None]
    if case["op"] == "layer":
        def adjoint(up):
            z = F.pad(up, (PAD, N - W - PAD, PAD, M - H - PAD))
            z[:, 0, 0] -= up.sum(dim=(1, 2))
            w = _convolve(z)[:, PAD:PAD + H + 1, PAD:PAD + W + 1]
            return w[:, :H, :W] - w[:, :H, 1:], w[:, :H, :W] - w[:, 1:, :W]

        ggx, ggy = _by_fields(adjoint, s["up"])
        return {"out": out, "grad_gx": ggx, "grad_gy": ggy}
    return out
