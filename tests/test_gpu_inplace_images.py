"""The uint8 in-place form on several images at once: interleaved stacks whose
images start on a store's boundary and off it, and the pre-process on enough
images that the form is taken (a few short rows stay on the FP32 forms)."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["bilinear", "bicubic"])
@pytest.mark.parametrize("C", [1, 2, 3, 4])
@pytest.mark.parametrize("W,Wo", [(62, 124), (100, 200), (250, 500), (90, 248), (300, 256)])
def test_interleaved_stacks(W, Wo, C, method):
    N, H, Ho = 3, 37, 74
    g = np.random.default_rng(W * C)
    x = torch.from_numpy(g.integers(0, 256, (N, H, W, C), dtype=np.uint8)).cuda()
    ref = torch.stack([rs.resize(t, (Ho, Wo), method, impl="tiled") for t in x])
    size = Ho * Wo * C
    for gap, off in ((0, 0), (16, 0), (1, 0), (6, 0), (16, 1), (48, 4)):   # bytes between images, before the first
        buf = torch.full((N * (size + gap) + 64,), 77, dtype=torch.uint8, device="cuda")
        y = torch.as_strided(buf, (N, Ho, Wo, C), (size + gap, Wo * C, C, 1), off)
        rs.resize(x, (Ho, Wo), method, impl="window", tile=(0, 4), out=y)
        assert torch.equal(y, ref), (gap, off)
        y.fill_(77)
        assert (buf == 77).all(), (gap, off)   # nothing written between the images
    assert rs.debug_fault() == 0


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("W,Wo", [(100, 256), (300, 512), (455, 455), (455, 456), (700, 455), (1024, 512), (9, 5),
                                  (130, 260), (650, 250), (515, 255)])
def test_normalize_stacks(W, Wo, dtype):
    mean, std = (123.675, 116.28, 103.53), (58.395, 57.12, 57.375)
    N = 48
    for C in (1, 3):
        for method, coord in (("bilinear", "half_pixel"), ("bicubic", "asymmetric")):
            Ho = 82 if Wo == 2 * W else 29
            g = np.random.default_rng(W)
            x = torch.from_numpy(g.integers(0, 256, (N, 41, W, C), dtype=np.uint8)).cuda()
            y = rs.resize_normalize(x, (Ho, Wo), method, mean[:C], std[:C], dtype=dtype, coord=coord)
            v = rs.resize(x.float(), (Ho, Wo), method, coord=coord, impl="tiled").double().permute(0, 3, 1, 2)
            sc = torch.tensor([np.float32(1) / np.float32(s) for s in std[:C]], device="cuda").double().view(1, C, 1, 1)
            bi = torch.tensor([-np.float32(m) / np.float32(s) for m, s in zip(mean, std)][:C], device="cuda").double()
            # one FP32 multiply-add of the FP32 value, then one rounding to the output type
            assert torch.equal(y, (v * sc + bi.view(1, C, 1, 1)).float().to(dtype))
    assert rs.debug_fault() == 0
