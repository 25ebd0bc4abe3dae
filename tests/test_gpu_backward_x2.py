"""The exact-x2 adjoint at the edges of its runs, warps, strips, chunks and
bands: bit for bit the two-pass kernels' results (the same sums in the same
order), under both maps it serves."""
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["bilinear", "bicubic"])
@pytest.mark.parametrize("coord", ["asymmetric", "half_pixel"])
@pytest.mark.parametrize("W", [2, 4, 6, 62, 64, 66, 130, 254, 256, 510, 512, 514, 1030])
def test_equals_two_pass(W, coord, method):
    g = torch.Generator(device="cuda").manual_seed(W)
    for H, planes in ((1, 1), (2, 3), (3, 2), (4, 1), (37, 2), (300, 1), (64, 40)):
        dy = torch.randn(1, planes, 2 * H, 2 * W, generator=g, device="cuda")
        for a in (-0.5, -0.75):
            x = rs.resize_backward(dy, (H, W), method, coord=coord, cubic_a=a)
            y = rs.resize_backward(dy, (H, W), method, coord=coord, cubic_a=a, impl="stream")
            assert torch.equal(x, y), (H, planes, a)
    assert rs.debug_fault() == 0
