"""The streaming antialias kernel at the bounds of what it holds: single output
rows of thousands of source rows (weights kept once instead of as pairs), one
output column's footprint wider than 128 threads own."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs
from oracle import oracle
from tests._parity import as_f64, check, to_storage

pytestmark = pytest.mark.gpu

NAMES = {1: "bilinear", 2: "bicubic"}


def image(H, W, C, dtype):
    g = np.random.default_rng(H * W)
    return to_storage(g.integers(0, 256, (H, W, C)).astype(np.float64), dtype).cuda()   # exact in every storage dtype


@pytest.mark.parametrize("H,W,C,Ho,Wo,dtype,method", [
    # rows: around and beyond what pairs leave room for
    (6700, 24, 3, 1, 3, "u8", 2), (7000, 64, 3, 1, 8, "u8", 2), (7500, 64, 1, 4, 8, "u8", 2), (8000, 1200, 3, 2, 120, "u8", 2),
    (9218, 1, 1, 1, 1, "u8", 2), (8015, 1, 4, 4, 12, "f16", 2), (8506, 12, 1, 4, 3, "f32", 2), (7413, 88, 4, 4, 39, "bf16", 2),
    (8000, 33, 3, 5, 7, "u8", 2), (9001, 40, 1, 3, 5, "u8", 1),
    # columns: FP32 footprints of 510 elements and more
    (1000, 200, 3, 3, 2, "f32", 1), (65, 207, 3, 1, 2, "f32", 1), (444, 206, 4, 20, 2, "f32", 1), (264, 882, 1, 1, 4, "f32", 1),
    (20, 129, 4, 1, 1, "f32", 1), (33, 510, 1, 5, 1, "f32", 2), (90, 1019, 1, 7, 1, "f16", 2), (31, 150, 4, 7, 1, "f32", 2),
    (100, 195, 3, 9, 2, "f32", 1)])
def test_footprints(H, W, C, Ho, Wo, dtype, method):
    x = image(H, W, C, dtype)
    ref = oracle.resize_aa(as_f64(x), Ho, Wo, method)
    for impl in ("stream", "auto"):
        y = rs.resize(x, (Ho, Wo), NAMES[method], antialias=True, impl=impl)
        check(y, ref, dtype, method, 255.0, f"{impl} {dtype} {H}x{W}x{C}->{Ho}x{Wo}")
    pad = torch.zeros(H, W * C + 3, dtype=x.dtype, device="cuda")   # any row alignment
    xp = pad[:, 1:1 + W * C].unflatten(1, (W, C))
    xp.copy_(x)
    assert torch.equal(rs.resize(xp, (Ho, Wo), NAMES[method], antialias=True, impl="stream"),
                       rs.resize(x, (Ho, Wo), NAMES[method], antialias=True, impl="stream"))
    assert rs.debug_fault() == 0


def test_preprocess_of_long_columns():
    mean, std = (123.675, 116.28, 103.53), (58.395, 57.12, 57.375)
    x = image(7000, 64, 3, "u8")
    y = rs.resize_normalize(x, (1, 8), "bicubic", mean, std, dtype=torch.float32, antialias=True)
    v = oracle.resize_aa(as_f64(x), 1, 8, 2)
    ref = ((v - np.array(mean)) / np.array(std)).transpose(2, 0, 1)
    assert np.abs(y.double().cpu().numpy() - ref).max() <= 1e-5 * 255 / min(std) + 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("H,W,C,Ho,Wo,dtype,method", [(756, 315, 3, 3, 1, "f32", 2), (1742, 209, 3, 13, 1, "f32", 2)])
def test_refused_as_before(H, W, C, Ho, Wo, dtype, method):
    """Beyond the form's range only what fits it as it is."""
    for impl in ("stream", "auto"):
        with pytest.raises(rs.ResampleError):
            rs.resize(image(H, W, C, dtype), (Ho, Wo), NAMES[method], antialias=True, impl=impl)
