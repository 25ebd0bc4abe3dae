"""Performance cases of the resampling library: what a user has it do, through
its public entry points, over the range of sizes it serves.

Kinds of case (case["kind"]):
  resize      one image or plane stack through resize(): uint8 interleaved
              images and float fields, nearest / bilinear / bicubic, with or
              without the antialias option
  train       ResizeFn on an FP32 NCHW tensor: the forward and its gradient
  preprocess  resize_normalize(): decoded uint8 frames to normalised planar
              network input, point-sampled or antialiased
  plan        BatchedPlan: a recorded ragged batch, replayed
  batch       resize_batched(): a ragged batch called once, work list and all

Outputs of the ragged kinds live in one buffer (each image's rows at a
256-byte aligned offset), as a serving program lays out its reply; run()
returns that buffer.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1001_1718_gb300 as rs

DTYPES = {"u8": torch.uint8, "f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
SIZE = {"u8": 1, "f16": 2, "bf16": 2, "f32": 4}
MEAN = (123.675, 116.28, 103.53)   # the usual image-network constants, in 0..255 units
STD = (58.395, 57.12, 57.375)


def listed():
    return [
        # The smallest call: a grey 512 x 512 image doubled; its time is the call and one short launch.
        dict(name="u8_512_bilinear_x2", kind="resize", dtype="u8", N=1, H=512, W=512, C=1, Ho=1024, Wo=1024,
             method="bilinear", coord="asymmetric", a=-0.5, antialias=False),
        # A large photograph doubled (the most common enlargement).
        dict(name="rgb4096_bicubic_x2", kind="resize", dtype="u8", N=1, H=4096, W=4096, C=3, Ho=8192, Wo=8192,
             method="bicubic", coord="asymmetric", a=-0.5, antialias=False),
        # The same photograph at a ratio that is no whole number, odd output sizes.
        dict(name="rgb4096_bicubic_x1.7", kind="resize", dtype="u8", N=1, H=4096, W=4096, C=3, Ho=6963, Wo=6963,
             method="bicubic", coord="asymmetric", a=-0.5, antialias=False),
        # The same photograph doubled without interpolation (label maps, previews): bytes moved.
        dict(name="rgb4096_nearest_x2", kind="resize", dtype="u8", N=1, H=4096, W=4096, C=3, Ho=8192, Wo=8192,
             method="nearest", coord="asymmetric", a=-0.5, antialias=False),
        # A scientific field in half precision, doubled: the largest float image.
        dict(name="field8192_bicubic_x2_f16", kind="resize", dtype="f16", N=1, H=8192, W=8192, C=1, Ho=16384,
             Wo=16384, method="bicubic", coord="asymmetric", a=-0.5, antialias=False),
        # A thumbnail of an odd-sized photograph with the antialias filter (16 taps an axis and more).
        dict(name="rgb4001x3003_thumb_aa", kind="resize", dtype="u8", N=1, H=3003, W=4001, C=3, Ho=683, Wo=910,
             method="bicubic", coord="half_pixel", a=-0.5, antialias=True),
        # Training: an enlarging layer, forward and backward.
        dict(name="train_32x3x512_bicubic_x2", kind="train", N=32, C=3, H=512, W=512, Ho=1024, Wo=1024,
             method="bicubic", coord="asymmetric", a=-0.5, antialias=False),
        # Training: a feature map enlarged between the levels of a pyramid, pixel centres
        # mapped as other frameworks do by default, sizes no multiple of 4.
        dict(name="train_8x64x90x130_half_pixel", kind="train", N=8, C=64, H=90, W=130, Ho=180, Wo=260,
             method="bilinear", coord="half_pixel", a=-0.5, antialias=False),
        # Network input from decoded square frames, halved.
        dict(name="pre_32x1024_to_512_f16", kind="preprocess", dtype="f16", N=32, H=1024, W=1024, C=3, Ho=512,
             Wo=512, method="bilinear", coord="asymmetric", a=-0.5, antialias=False),
        # Network input from video frames with the antialias filter.
        dict(name="pre_16x1080p_to_256x455_aa", kind="preprocess", dtype="f16", N=16, H=1080, W=1920, C=3, Ho=256,
             Wo=455, method="bilinear", coord="asymmetric", a=-0.5, antialias=True),
        # A request of a few images of uneven sizes, called once: the work list is part of the call.
        dict(name="batch24_request", kind="batch", n=24, lo=64, hi=1024, smin=0.5, smax=4.0, C=3, sizes=11,
             coord="half_pixel", a=-0.75, antialias=False),
        # The large ragged batch, replayed from its plan.
        dict(name="batch256_plan", kind="plan", n=256, lo=64, hi=2048, smin=0.5, smax=4.0, C=3, sizes=4,
             coord="asymmetric", a=-0.5, antialias=False),
    ]


# ---------------------------------------------------------------------------
# Drawn cases

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _scaled(n, s):
    return max(1, int(n * s))


def draw(rng):
    coord = rng.choice(["asymmetric", "half_pixel", "align_corners"])
    a = rng.choice([-0.5, -0.75])
    kind = rng.choice(["resize", "resize", "resize", "train", "preprocess", "plan", "batch"])
    if kind in ("plan", "batch"):
        return dict(kind=kind, n=_log(rng, 8, 64), lo=64, hi=rng.choice([640, 1024, 2048]), smin=0.5, smax=4.0,
                    C=rng.choice([1, 3, 3, 4]), sizes=rng.randrange(1 << 20), coord=coord, a=a,
                    antialias=rng.random() < 0.25)
    if kind == "preprocess":
        aa = rng.random() < 0.5
        N, H, W = _log(rng, 1, 32), _log(rng, 160, 1440), _log(rng, 160, 1920)
        s = rng.uniform(0.15, 1.0) if aa else rng.uniform(0.4, 2.0)
        return dict(kind=kind, dtype=rng.choice(["f16", "bf16", "f32"]), N=N, H=H, W=W, C=3, Ho=_scaled(H, s),
                    Wo=_scaled(W, s), method=rng.choice(["bilinear", "bicubic"]), coord=coord, a=a, antialias=aa)
    if kind == "train":
        H, W, C = _log(rng, 24, 512), _log(rng, 24, 512), rng.choice([1, 3, 16, 64])
        N = max(1, min(32, 24_000_000 // (C * H * W)))
        s = 2.0 if rng.random() < 0.4 else rng.uniform(0.35, 2.6)
        return dict(kind=kind, N=N, C=C, H=H, W=W, Ho=_scaled(H, s), Wo=_scaled(W, s),
                    method=rng.choice(["bilinear", "bicubic"]), coord=coord, a=a,
                    antialias=s < 1 and rng.random() < 0.5)
    dtype = rng.choice(["u8", "u8", "f16", "bf16", "f32"])
    C = rng.choice([1, 3, 3, 4]) if dtype == "u8" else 1
    H, W = _log(rng, 64, 4200), _log(rng, 64, 4200)
    aa = rng.random() < 0.25
    s = 2.0 if rng.random() < 0.25 else rng.uniform(0.12, 1.0) if aa else rng.uniform(0.4, 3.5)
    aa = aa and s < 1
    method = rng.choice(["bilinear", "bicubic"] if aa else ["nearest", "bilinear", "bilinear", "bicubic", "bicubic"])
    return dict(kind=kind, dtype=dtype, N=1, H=H, W=W, C=C, Ho=_scaled(H, s), Wo=_scaled(W, s), method=method,
                coord=coord, a=a, antialias=aa)


# ---------------------------------------------------------------------------
# Inputs

def _photo(g, N, H, W, C):
    """(N, H, W, C) uint8: a smooth field of Gaussian blobs plus noise, as photographs vary."""
    dev = g.device
    nb = 12
    amp = torch.rand(nb, C, generator=g, device=dev) * 192 - 96
    sig = torch.rand(nb, 1, generator=g, device=dev) * 0.3 + 0.05
    cy, cx = torch.rand(nb, 1, generator=g, device=dev), torch.rand(nb, 1, generator=g, device=dev)
    y = torch.linspace(0, 1, H, device=dev)[None]
    x = torch.linspace(0, 1, W, device=dev)[None]
    gy = torch.exp(-((y - cy) / sig) ** 2 / 2)
    gx = torch.exp(-((x - cx) / sig) ** 2 / 2)
    field = gy.t() @ (gx[:, :, None] * amp[:, None, :]).reshape(nb, W * C) + 128
    out = torch.empty(N, H, W * C, dtype=torch.uint8, device=dev)
    for k in range(N):
        noise = torch.rand(H, W * C, generator=g, device=dev).mul_(16).sub_(8)
        out[k] = noise.add_(field).round_().clamp_(0, 255)
    return out.view(N, H, W, C)


def _ragged(case):
    """Sizes, scales and methods of a ragged batch, from the case alone: (H, W, Ho, Wo, method)."""
    g = np.random.Generator(np.random.PCG64(case["sizes"]))
    n = case["n"]
    H = g.integers(case["lo"], case["hi"] + 1, size=n)
    W = g.integers(case["lo"], case["hi"] + 1, size=n)
    s = g.uniform(case["smin"], case["smax"], size=n)
    return [(int(h), int(w), _scaled(int(h), float(f)), _scaled(int(w), float(f)),
             "bicubic" if k % 2 else "bilinear") for k, (h, w, f) in enumerate(zip(H, W, s))]


def _sources(case, seed):
    """The case's input tensors (the incoming gradient of a training case last)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind in ("plan", "batch"):
        return [_photo(g, 1, h, w, case["C"])[0] for h, w, _, _, _ in _ragged(case)]
    N, C, H, W = case["N"], case["C"], case["H"], case["W"]
    if kind == "train":
        return [torch.randn(N, C, H, W, generator=g, device="cuda"),
                torch.randn(N, C, case["Ho"], case["Wo"], generator=g, device="cuda")]
    if kind == "preprocess" or case["dtype"] == "u8":
        x = _photo(g, N, H, W, C)
        return [x[0] if kind == "resize" else x]
    y = torch.linspace(0, 6.0, H, device="cuda")[:, None]
    x = torch.linspace(0, 9.0, W, device="cuda")[None]
    field = torch.rand(H, W, generator=g, device="cuda").add_(0.5 * torch.sin(y) * torch.cos(x))
    return [field.to(DTYPES[case["dtype"]])]


def _arena(case):
    """Offsets of the ragged outputs in one buffer and its length."""
    at, offs = 0, []
    for _, _, ho, wo, _ in _ragged(case):
        offs.append(at)
        at += -(-ho * wo * case["C"] // 256) * 256
    return offs, at


def prepare(case, seed):
    src = _sources(case, seed)
    state = dict(case=case, src=src)
    if case["kind"] in ("plan", "batch"):
        offs, total = _arena(case)
        reply = torch.zeros(total, dtype=torch.uint8, device="cuda")
        C = case["C"]
        state["reply"] = reply
        state["outs"] = [reply[o:o + ho * wo * C].view(ho, wo, C)
                         for o, (_, _, ho, wo, _) in zip(offs, _ragged(case))]
        state["sizes"] = [(ho, wo) for _, _, ho, wo, _ in _ragged(case)]
        state["methods"] = [m for *_, m in _ragged(case)]
        if case["kind"] == "plan":
            state["plan"] = rs.BatchedPlan(src, state["outs"], state["methods"], coord=case["coord"],
                                           cubic_a=case["a"], antialias=case["antialias"])
    elif case["kind"] == "train":
        src[0].requires_grad_(True)
    return state


def run(state):
    case, src = state["case"], state["src"]
    kind = case["kind"]
    if kind == "plan":
        state["plan"].launch()
        return state["reply"]
    if kind == "batch":
        rs.resize_batched(src, state["sizes"], state["methods"], coord=case["coord"], cubic_a=case["a"],
                          outs=state["outs"], antialias=case["antialias"])
        return state["reply"]
    size = (case["Ho"], case["Wo"])
    if kind == "train":
        x, g = src
        y = rs.ResizeFn.apply(x, size, case["method"], case["coord"], case["a"], case["antialias"])
        (gx,) = torch.autograd.grad(y, x, g)
        return [y, gx]
    if kind == "preprocess":
        return rs.resize_normalize(src[0], size, case["method"], MEAN, STD, dtype=DTYPES[case["dtype"]],
                                   coord=case["coord"], cubic_a=case["a"], antialias=case["antialias"])
    return rs.resize(src[0], size, case["method"], coord=case["coord"], cubic_a=case["a"],
                     antialias=case["antialias"])


# ---------------------------------------------------------------------------
# Work: each input read once, each output written once; the multiply-adds of
# the separable form (horizontal taps per source row used, vertical taps per output).

def _axis_taps(n, m, method, antialias):
    if method == "nearest":
        return 0
    k = 2 if method == "bilinear" else 4
    return k * max(n / m, 1.0) if antialias else k


def _flops(case, H, W, Ho, Wo, method, planes):
    ky, kx = (_axis_taps(n, m, method, case["antialias"]) for n, m in ((H, Ho), (W, Wo)))
    return 2.0 * planes * (min(H, Ho * ky) * Wo * kx + Ho * Wo * ky)


def work(case):
    kind = case["kind"]
    if kind in ("plan", "batch"):
        C = case["C"]
        images = _ragged(case)
        return {"bytes": sum((h * w + ho * wo) * C for h, w, ho, wo, _ in images),
                "flops": sum(_flops(case, h, w, ho, wo, m, C) for h, w, ho, wo, m in images)}
    H, W, Ho, Wo, planes = case["H"], case["W"], case["Ho"], case["Wo"], case["N"] * case["C"]
    f = _flops(case, H, W, Ho, Wo, case["method"], planes)
    if kind == "train":
        return {"bytes": 2 * 4 * planes * (H * W + Ho * Wo), "flops": 2 * f}
    si = 1 if kind == "preprocess" else SIZE[case["dtype"]]
    return {"bytes": planes * (H * W * si + Ho * Wo * SIZE[case["dtype"]]), "flops": f}


# ---------------------------------------------------------------------------
# The same results in 64 bits, by plain torch

def _keys(u, a):
    u = u.abs()
    near = ((a + 2) * u - (a + 3)) * u * u + 1
    far = ((a * u - 5 * a) * u + 8 * a) * u - 4 * a
    return torch.where(u <= 1, near, torch.where(u < 2, far, torch.zeros_like(u)))


def _axis(n, m, case, method):
    """Taps of an axis of m outputs from n samples: indices and weights, (m, K)."""
    j = torch.arange(m, device="cuda", dtype=torch.int64)
    a = case["a"]
    if case["antialias"]:
        R, F = (1 if method == "bilinear" else 2), max(n, m)
        c = (2 * j + 1) * n   # centre in units of 1 / (2 m)
        lo = torch.div(c - 2 * R * F + m, 2 * m, rounding_mode="floor")
        hi = torch.div(c + 2 * R * F + m, 2 * m, rounding_mode="floor")
        i = lo[:, None] + torch.arange(int((hi - lo).max()), device="cuda")
        u = ((2 * i + 1) * m - c[:, None]).double() / (2 * F)
        w = (1 - u.abs()).clamp(min=0) if method == "bilinear" else _keys(u, a)
        w = torch.where((i >= 0) & (i < n) & (i < hi[:, None]), w, torch.zeros_like(w))
        return i.clamp(0, n - 1), w / w.sum(1, keepdim=True)
    if case["coord"] == "asymmetric":
        num, den = j * n, m
    elif case["coord"] == "half_pixel":
        num, den = (2 * j + 1) * n - m, 2 * m
    else:
        num, den = j * (n - 1), max(m - 1, 1)
    if method == "nearest":
        if case["coord"] != "asymmetric":
            num, den = 2 * num + den, 2 * den
        return torch.div(num, den, rounding_mode="floor").clamp(0, n - 1)[:, None], torch.ones(m, 1, device="cuda").double()
    i0 = torch.div(num, den, rounding_mode="floor")
    t = (num - i0 * den).double() / den
    if method == "bilinear":
        return torch.stack([i0, i0 + 1], 1).clamp(0, n - 1), torch.stack([1 - t, t], 1)
    k = torch.arange(-1, 3, device="cuda")
    return (i0[:, None] + k).clamp(0, n - 1), _keys(t[:, None] - k, a)


def _apply(x, dim, idx, w):
    shape = [1] * x.dim()
    shape[dim] = -1
    out = 0.0
    for k in range(idx.shape[1]):
        out = out + x.index_select(dim, idx[:, k]) * w[:, k].view(shape)
    return out


def _transpose(y, dim, idx, w, n):
    shape = list(y.shape)
    shape[dim] = n
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    view = [1] * y.dim()
    view[dim] = -1
    for k in range(idx.shape[1]):
        out.index_add_(dim, idx[:, k], y * w[:, k].view(view))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("plan", "batch"):
        return None   # bytes: nothing but whole numbers comes back
    src = _sources(case, seed)
    ay = _axis(case["H"], case["Ho"], case, case["method"])
    ax = _axis(case["W"], case["Wo"], case, case["method"])
    x = src[0].double()
    if kind == "train":
        y = _apply(_apply(x, 3, *ax), 2, *ay)
        gx = _transpose(_transpose(src[1].double(), 2, *ay, case["H"]), 3, *ax, case["W"])
        return [y, gx]
    if kind == "preprocess":
        x = x.permute(0, 3, 1, 2)
        y = _apply(_apply(x, 3, *ax), 2, *ay)
        mean, std = (torch.tensor(v, device="cuda").double().view(1, 3, 1, 1) for v in (MEAN, STD))
        return (y - mean) / std
    y = _apply(_apply(x, 1, *ax), 0, *ay)
    return y.clamp(0, 255).round().to(torch.uint8) if case["dtype"] == "u8" else y
