"""The register-window form that reads uint8 sources in place: byte for byte the
tiled kernel's results (the library's forward kernels share one order of
operations) at the edges of its ratio ranges, warps, strips and store forms,
and nothing written outside the image."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu

COORDS = ["asymmetric", "half_pixel", "align_corners"]


def image(seed, H, W, C, pad, off):
    """(H, W, C) uint8 view of a buffer, rows W C + pad bytes apart, starting at byte off."""
    g = np.random.default_rng(seed)
    buf = torch.from_numpy(g.integers(0, 256, H * (W * C + pad) + off + 16, dtype=np.uint8)).cuda()
    return buf, buf[off:off + H * (W * C + pad)].view(H, W * C + pad)[:, :W * C].unflatten(1, (W, C))


def check(H, W, C, Ho, Wo, method, coord, a=-0.5, pad=0, off=0):
    _, x = image(H * 31 + W, H, W, C, pad, off)
    buf, y = image(7, Ho, Wo, C, pad, off)
    before = buf.clone()
    ref = rs.resize(x.contiguous(), (Ho, Wo), method, coord=coord, cubic_a=a, impl="tiled")
    # (beyond two source pixels per output pixel the default chunk of 8 rows is
    # refused: the general form's footprint rule)
    rs.resize(x, (Ho, Wo), method, coord=coord, cubic_a=a, impl="window", tile=(0, 4) if W > 2 * Wo else None, out=y)
    assert rs.debug_fault() == 0
    assert torch.equal(y, ref)
    y.copy_(before[off:off + Ho * (Wo * C + pad)].view(Ho, Wo * C + pad)[:, :Wo * C].unflatten(1, (Wo, C)))
    assert torch.equal(buf, before), "bytes outside the image changed"


# Output widths around a run (4), a warp (124 / 128) and a strip (496 / 512);
# odd pitches and offsets take every phase of the row's words.
@pytest.mark.parametrize("method", ["bilinear", "bicubic"])
@pytest.mark.parametrize("Wo", [1, 2, 3, 4, 5, 7, 8, 123, 124, 125, 128, 129, 495, 496, 497, 500, 512, 513, 997])
def test_widths(Wo, method):
    for k, C in enumerate((1, 2, 3, 4)):
        W = max(1, int(Wo / 1.37))
        check(23, W, C, 37, Wo, method, COORDS[k % 3], pad=0)
        check(23, W, C, 37, Wo, method, COORDS[(k + 1) % 3], pad=k + 1, off=k + 3)


# Ratios at and around the bounds of the four ratio ranges (1/2, 1, 2, 3 source
# pixels per output pixel), and vertical ratios of their own.
@pytest.mark.parametrize("coord", COORDS)
@pytest.mark.parametrize("W,Wo", [(100, 401), (100, 400), (150, 449), (200, 400), (201, 401), (200, 399), (256, 384),
                                  (400, 401), (300, 300), (401, 400), (600, 400), (799, 400), (800, 400), (801, 401),
                                  (1023, 512), (1025, 512), (1201, 400), (1199, 400), (900, 300)])
def test_ratios(W, Wo, coord):
    for method, a in (("bilinear", -0.5), ("bicubic", -0.5), ("bicubic", -0.75)):
        for H, Ho in ((37, 90), (90, 37), (1, 5), (5, 1), (300, 300)):
            check(H, W, 3, Ho, Wo, method, coord, a)


# The exact x2 form: runs, warps and strips of doubled widths, one source row
# to several bands.
@pytest.mark.parametrize("method", ["bilinear", "bicubic"])
@pytest.mark.parametrize("W", [1, 2, 3, 31, 62, 63, 64, 124, 247, 248, 249, 256, 257, 500])
def test_x2(W, method):
    for k, C in enumerate((1, 2, 3, 4)):
        for H in (1, 2, 37, 300):
            check(H, W, C, 2 * H, 2 * W, method, "asymmetric")
        check(37, W, C, 74, 2 * W, method, "asymmetric", a=-0.75, pad=k + 1, off=k + 3)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("W,Wo", [(100, 257), (300, 512), (455, 455), (700, 455), (1024, 512), (9, 5), (130, 260), (63, 126), (650, 250), (515, 255)])
def test_normalize(W, Wo, dtype):
    mean, std = (123.675, 116.28, 103.53), (58.395, 57.12, 57.375)
    for C in (1, 3):
        for method, coord in (("bilinear", "half_pixel"), ("bicubic", "asymmetric")):
            _, x = image(W, 41, W, C, 5, 1)
            x2 = torch.stack([x, x.flip(0)])
            Ho = 82 if Wo == 2 * W else 29
            y = rs.resize_normalize(x2, (Ho, Wo), method, mean[:C], std[:C], dtype=dtype, coord=coord)
            v = rs.resize(x2.float(), (Ho, Wo), method, coord=coord, impl="tiled").double().permute(0, 3, 1, 2)
            sc = torch.tensor([np.float32(1) / np.float32(s) for s in std[:C]], device="cuda").double().view(1, C, 1, 1)
            bi = torch.tensor([-np.float32(m) / np.float32(s) for m, s in zip(mean, std)][:C], device="cuda").double()
            # one FP32 multiply-add of the FP32 value, then one rounding to the output type
            assert torch.equal(y, (v * sc + bi.view(1, C, 1, 1)).float().to(dtype))
    assert rs.debug_fault() == 0
