"""Calls whose marshalled arguments are kept by value: the same call gives the
same answer whatever calls came before it."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [0.0, -0.0])
def test_zeros_of_either_sign(first):
    """y = x / std - mean / std in one multiply-add: with x = 0 and std = -1
    the product is -0 and the sum takes the sign of mean's zero."""
    rs._CALLS.clear()
    x = torch.zeros(40, 50, 1, dtype=torch.uint8, device="cuda")
    for mean in (first, -first, first):
        y = rs.resize_normalize(x, (30, 40), "bilinear", (mean,), (-1.0,), dtype=torch.float32)
        assert (torch.signbit(y) == bool(np.signbit(np.float32(mean)))).all()
    xf = torch.full((1, 8, 8), -0.0, device="cuda")   # the outer taps' weights are zeros of a's sign
    got = {}
    for a in (first, -first, first):
        y = rs.resize(xf, (16, 16), "bicubic", layout="nchw", cubic_a=a, impl="tiled")
        sign = torch.signbit(y)
        assert str(a) not in got or torch.equal(got[str(a)], sign)
        got[str(a)] = sign


def test_batch_refusals_do_not_depend_on_earlier_batches():
    """The workspace query refuses a bicubic image of 1/30 (its point-sampled
    tiles do not fit), antialiased or not, first or after other batches."""
    small = torch.zeros(20, 20, 3, dtype=torch.uint8, device="cuda")
    wide = torch.zeros(40, 1200, 3, dtype=torch.uint8, device="cuda")
    rs._CALLS.clear()
    for _ in range(2):
        for aa in (False, True):
            with pytest.raises(rs.ResampleError):
                rs.resize_batched([wide], [(20, 40)], ["bicubic"], antialias=aa)
        rs.resize_batched([small], [(30, 30)], ["bilinear"])


@pytest.mark.parametrize("C", [1, 2, 3, 4])
@pytest.mark.parametrize("method", ["nearest", "bilinear", "bicubic"])
def test_rows_of_a_24th_always_fit(C, method):
    """The ratio down to which the query's answer is kept."""
    for Wo in (1, 7, 64, 600):
        x = torch.zeros(9, 24 * Wo, C, dtype=torch.uint8, device="cuda")
        y = torch.zeros(5, Wo, C, dtype=torch.uint8, device="cuda")
        assert rs.batched_workspace_bytes([x], [y], [method]) > 0
        rs.resize_batched([x], [(5, Wo)], [method], outs=[y])
    assert rs.debug_fault() == 0
