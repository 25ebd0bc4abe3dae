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
