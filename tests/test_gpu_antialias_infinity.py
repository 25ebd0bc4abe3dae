"""An infinity or a NaN in an antialiased float image reaches the outputs whose
taps include it and no others, wherever the streaming kernel's bands begin."""
import pytest
import torch

import paper_1001_1718_gb300 as rs

pytestmark = pytest.mark.gpu


def taps(j, n, m, R):
    F, a = max(n, m), (2 * j + 1) * n + m
    return max((a - 2 * R * F) // (2 * m), 0), min((a + 2 * R * F) // (2 * m), n)


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("method,H,Ho", [("bilinear", 300, 50), ("bicubic", 300, 50), ("bicubic", 211, 97), ("bilinear", 97, 6)])
def test_one_in_every_row(method, H, Ho, dtype):
    """Image n of a stack holds one in row n (so many images that a block's
    band has several output rows)."""
    W, Wo, R, N = 90, 12, 1 if method == "bilinear" else 2, max(H, 200)
    g = torch.Generator(device="cuda").manual_seed(H)
    x = torch.rand((N, 1, H, W), generator=g, device="cuda").to(dtype)
    ref = rs.resize(x, (Ho, Wo), method, layout="nchw", antialias=True, impl="stream")
    reach = torch.zeros((N, 1, Ho, Wo), dtype=torch.bool)
    cols = [taps(j, W, Wo, R) for j in range(Wo)]
    for n in range(N):
        y, px = n % H, 7 * n % W
        x[n, 0, y, px] = float("inf") if n % 2 else float("nan")
        for i in range(Ho):
            a, b = taps(i, H, Ho, R)
            if a <= y < b:
                for j, (c, d) in enumerate(cols):
                    reach[n, 0, i, j] = c <= px < d
    got = rs.resize(x, (Ho, Wo), method, layout="nchw", antialias=True, impl="stream")
    out = ~reach.cuda()
    bad = (got != ref) & out
    assert not bad.any(), f"{int(bad.sum())} outputs, output rows {sorted(set(bad.nonzero()[:, 2].tolist()))}"
    assert not torch.isfinite(got[~out]).all()
    assert rs.debug_fault() == 0
