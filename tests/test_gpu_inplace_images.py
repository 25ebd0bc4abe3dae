"""The uint8 in-place form on several images at once: interleaved stacks whose
images start on a store's boundary and off it."""
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
