"""The narrower tiles of launches with few tiles: an image's outputs do not
depend on the tile width (each is one chain over the same K-blocks), so the
first images of a batch large enough for full-width tiles must come out bit
for bit as they do alone, where the tiles are 64 or 128 wide; and the fused
statistics of the small launch must close to the same BatchNorm."""
import numpy as np
import pytest
import torch

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300 import synthetic as syn
from gpu_util import dev, empty16, host

pytestmark = pytest.mark.gpu


# h, w, c, k, r, stride; images alone (tiles fit the SMs) and in the large batch (they do not)
CASES = [(14, 14, 128, 256, 1, 1, 3, 80), (14, 14, 64, 320, 3, 1, 2, 60), (16, 16, 256, 192, 3, 2, 5, 200),
         (7, 7, 512, 512, 3, 1, 9, 500), (9, 11, 64, 576, 1, 2, 7, 250), (1, 1, 128, 1000, 1, 1, 130, 8000)]


@pytest.mark.parametrize("h,w,c,k,r,st,small,large", CASES)
def test_tile_width(h, w, c, k, r, st, small, large):
    g = torch.Generator(device="cuda").manual_seed(5)
    p, q = (h + 2 * (r // 2) - r) // st + 1, (w + 2 * (r // 2) - r) // st + 1
    f = lambda *s: torch.randn(s, device="cuda", generator=g).to(torch.float16)
    x, dy, wt = f(large, h, w, c), f(large, p, q, k), f(k, r, r, c)
    out = []
    for n in (small, large):
        d = pf16.conv_desc(n, h, w, c, k, r, r, st, r // 2)
        y, dx = torch.zeros_like(dy[:n]), torch.zeros_like(x[:n])
        pf16.conv_fwd(d, x, wt, y)
        pf16.conv_dgrad(d, dy, wt, dx)
        out.append((y, dx))
    assert pf16.sync_status() == 0
    for a, b in zip(*out):
        assert torch.equal(a.view(torch.int16), b[:small].view(torch.int16))


@pytest.mark.parametrize("n,h,c,k,r", [(2, 14, 64, 256, 1), (1, 9, 64, 192, 3)])
def test_statistics_slots(n, h, c, k, r):
    """Narrow tiles: each M tile's slot covers every channel with its row count."""
    d = pf16.conv_desc(n, h, h, c, k, r, r, 1, r // 2)
    x = dev(syn.normal_f16(42, (n, h, h, c)))
    w = dev(syn.he_normal_f16(43, k, r, r, c))
    y, stats = empty16(n * h * h * k), torch.zeros(pf16.conv_bnstats_size(d), dtype=torch.uint8, device="cuda")
    pf16.conv_fwd_bnstats(d, x, w, y, stats)
    assert pf16.sync_status() == 0
    raw = stats.cpu().numpy()
    slots = int(raw[:4].view(np.int32)[0])
    rows = n * h * h
    assert slots == (rows + 127) // 128
    mean = raw[256:256 + 256 * k * 2].view(np.float16).reshape(256, k)[:slots].astype(np.float64)
    v = host(y).view(np.float16).reshape(rows, k).astype(np.float64)
    for s in range(slots):
        blk = v[128 * s:128 * (s + 1)]
        # halving trees of depth 7 over the slot's rows (a ragged leaf is rescaled: one rounding more)
        tol = 12 * 2.0 ** -11 * np.abs(blk).max(0) + 2.0 ** -24
        assert np.all(np.abs(mean[s] - blk.mean(0)) <= tol)
