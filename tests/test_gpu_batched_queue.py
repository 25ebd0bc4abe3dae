"""The ragged batch's item queue and work list at their edges: items that take
all of a block's shared memory, lists around the upload's pieces, calls back to
back on one workspace. Every image equals its single-image call bit for bit."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu


def image(g, H, W, C, dtype=torch.uint8):
    x = torch.from_numpy(g.integers(0, 256, (H, W, C), dtype=np.uint8)).cuda()
    return x if dtype == torch.uint8 else x.to(dtype)


# Sizes whose tiles need exactly what a block may have (232448 bytes of shared
# memory), and 8 bytes less: many-tap antialias tiles, and point-sampled tiles.
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("H,W,C,Ho,Wo,method,aa", [(352, 707, 4, 32, 64, "bilinear", True), (568, 1154, 4, 32, 64, "bilinear", True),
                                                   (612, 819, 4, 48, 64, "bilinear", True), (64, 347, 1, 64, 16, "bilinear", False),
                                                   (64, 347, 1, 64, 16, "bicubic", False), (64, 1388, 1, 64, 64, "bilinear", False)])
def test_items_of_all_shared_memory(H, W, C, Ho, Wo, method, aa, dtype):
    x = image(np.random.default_rng(H + W), H, W, C, dtype)
    ref = rs.resize(x, (Ho, Wo), method, antialias=aa, impl="tiled")
    y, = rs.resize_batched([x], [(Ho, Wo)], [method], antialias=aa, impl="tiled")
    assert torch.equal(y, ref)
    y.zero_()
    plan = rs.BatchedPlan([x], [y], [method], antialias=aa, impl="tiled")
    for _ in range(2):
        plan.launch()
    assert torch.equal(y, ref)
    assert rs.debug_fault() == 0
