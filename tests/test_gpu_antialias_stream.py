"""The vertical-first streaming antialias kernel at the edges of its row groups
(4 output rows), bands, tiles and source alignments, against the FP64
definition; a pitched source takes the form for any row alignment and must
equal the aligned one bit for bit."""
import numpy as np
import pytest
import torch

import paper_1001_1718_gb300 as rs
from oracle import oracle
from tests._parity import as_f64, check, to_storage

pytestmark = pytest.mark.gpu

NAMES = {1: "bilinear", 2: "bicubic"}


@pytest.mark.parametrize("dtype", ["u8", "f16", "bf16", "f32"])
@pytest.mark.parametrize("H,W,C,Ho,Wo", [(40, 50, 3, 1, 1), (41, 33, 1, 2, 9), (90, 64, 4, 3, 7), (64, 129, 2, 5, 11),
                                         (200, 341, 3, 6, 76), (203, 400, 3, 47, 77), (120, 120, 3, 120, 20),
                                         (257, 1100, 1, 31, 250), (65, 8, 3, 13, 40)])
def test_edges(H, W, C, Ho, Wo, dtype):
    g = np.random.default_rng(H * W)
    x64 = g.integers(0, 256, (H, W, C)).astype(np.float64)   # exact in every storage dtype
    t = to_storage(x64, dtype).cuda()
    pad = torch.zeros(H, W * C + 3, dtype=t.dtype, device="cuda")
    xp = pad[:, 1:1 + W * C].unflatten(1, (W, C))
    xp.copy_(t)
    for method in (1, 2):
        y = rs.resize(t, (Ho, Wo), NAMES[method], antialias=True, impl="stream")
        yp = rs.resize(xp, (Ho, Wo), NAMES[method], antialias=True, impl="stream")
        check(y, oracle.resize_aa(as_f64(t), Ho, Wo, method), dtype, method, 255.0, f"{dtype} {H}x{W}x{C}->{Ho}x{Wo}")
        assert torch.equal(y, yp)
    assert rs.debug_fault() == 0
