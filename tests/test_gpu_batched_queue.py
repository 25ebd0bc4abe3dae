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


def ragged(seed, n, lo, hi, channels=(1, 2, 3, 4), smin=0.3, smax=3.0):
    g = np.random.default_rng(seed)
    xs, sizes, methods = [], [], []
    for k in range(n):
        H, W = (int(v) for v in g.integers(lo, hi + 1, 2))
        xs.append(image(g, H, W, channels[k % len(channels)]))
        sizes.append((max(1, int(H * g.uniform(smin, smax))), max(1, int(W * g.uniform(smin, smax)))))
        methods.append(("bilinear", "bicubic", "nearest", "bicubic")[k * 7 % 4])
    return xs, sizes, methods


def singles(xs, sizes, methods):
    return [rs.resize(x, s, m, impl="auto" if m == "nearest" else "tiled") for x, s, m in zip(xs, sizes, methods)]


# Work lists of one piece (up to 97 images), two (up to 200) and of a copy.
@pytest.mark.parametrize("n", [1, 97, 98, 150, 200, 201, 260])
def test_list_lengths(n):
    xs, sizes, methods = ragged(n, n, 5, 24)
    for y, r in zip(rs.resize_batched(xs, sizes, methods), singles(xs, sizes, methods)):
        assert torch.equal(y, r)
    assert rs.debug_fault() == 0


def test_calls_back_to_back_on_one_workspace():
    """Each call's list overwrites the one before in stream order: no wait
    between the calls, classes of all kinds, launches that overlap."""
    calls = [ragged(100 + k, (3, 40, 9, 120, 24)[k % 5], 8, 160) for k in range(10)]
    size = max(rs.batched_workspace_bytes(xs, [x.new_empty((*s, x.shape[2])) for x, s in zip(xs, sizes)], methods)
               for xs, sizes, methods in calls)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    refs = [singles(*c) for c in calls]
    torch.cuda.synchronize()
    for _ in range(3):
        got = [rs.resize_batched(*c, workspace=ws) for c in calls]
        torch.cuda.synchronize()
        for outs, ref in zip(got, refs):
            assert all(torch.equal(y, r) for y, r in zip(outs, ref))
    assert rs.debug_fault() == 0


@pytest.mark.parametrize("channels", [(3,), (1, 2, 3, 4)])
@pytest.mark.parametrize("n,lo,hi", [(3, 20, 60), (30, 20, 90), (60, 300, 700)])
def test_ratios_on_both_sides_of_two(n, lo, hi, channels):
    """uint8 images read in place (up to two source pixels per output pixel) and
    not, in one batch; few small images of all channel counts are not at all."""
    xs, sizes, methods = ragged(n + lo, n, lo, hi, channels, 0.35, 2.5)
    ref = singles(xs, sizes, methods)
    outs = rs.resize_batched(xs, sizes, methods)
    assert all(torch.equal(y, r) for y, r in zip(outs, ref))
    plan = rs.BatchedPlan(xs, outs, methods)
    for stream in (torch.cuda.Stream(), torch.cuda.Stream()):   # replays in turn on other streams
        for y in outs:
            y.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            plan.launch(stream.cuda_stream)
        torch.cuda.synchronize()
        assert all(torch.equal(y, r) for y, r in zip(outs, ref))
    assert rs.debug_fault() == 0
