"""The stem's convolution over many tiles per CTA (statistics by their own warps,
double staging): output and BatchNorm as for one of few, at the three padded row
widths, with full rows of 128 and with ragged CTA shares.  And its weight
gradient, whose windows run past the last column, exactly, on values whose sums
FP16 holds."""
import pytest
import torch
import torch.nn.functional as F

import test_gpu_convbn as convbn
from paper_1911_07384_gb300 import pf16
from gpu_util import workspace

pytestmark = pytest.mark.gpu

# tiles of 128 padded pixels: 1,400 (rows of 32), 1,280 (64), 1,250 (128, Q + 3 = 128)
STATS = [(200, 56, 56), (80, 64, 64), (10, 250, 250)]


@pytest.mark.parametrize("n,h,w", STATS)
def test_statistics(orc, n, h, w):
    convbn.test_conv_fwd_bnstats_then_bn(orc, (n, h, w, 3, 64, 7, 7, 2, 3))


@pytest.mark.parametrize("n,h,w", [(41, 250, 246), (350, 64, 58)])
def test_double_staging(n, h, w):
    """No statistics: the images of a large batch as in a batch of two."""
    g = torch.Generator(device="cuda").manual_seed(8)
    x = torch.randn((n, h, w, 3), device="cuda", generator=g).half()
    wt = (torch.randn((64, 7, 7, 3), device="cuda", generator=g) / 12).half()
    out = []
    for m in (n, 2):
        d = pf16.conv_desc(m, h, w, 3, 64, 7, 7, 2, 3)
        y = torch.zeros((m, (h + 1) // 2, (w + 1) // 2, 64), device="cuda", dtype=torch.float16)
        pf16.conv_fwd(d, x[n - m:].clone(), wt, y, workspace(pf16.conv_workspace_size(d, pf16.PF16_PASS_FWD)))
        out.append(y)
    assert pf16.sync_status() == 0
    assert torch.equal(out[0][n - 2:], out[1])


@pytest.mark.parametrize("n,h,w", [(3, 250, 250), (5, 20, 249), (2, 9, 11)])
def test_weight_gradient_exact(n, h, w):
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randint(-1, 2, (n, h, w, 3), device="cuda", generator=g).half()
    p, q = (h + 1) // 2, (w + 1) // 2
    dy = torch.randint(-1, 2, (n, p, q, 64), device="cuda", generator=g).half()
    dy *= torch.rand((n, p, q, 64), device="cuda", generator=g) < 0.02  # every partial sum below 2,048
    d = pf16.conv_desc(n, h, w, 3, 64, 7, 7, 2, 3)
    dw = torch.zeros((64, 7, 7, 3), device="cuda", dtype=torch.float16)
    pf16.conv_wgrad(d, x, dy, dw, workspace(pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD)))
    assert pf16.sync_status() == 0
    cols = F.unfold(x.cpu().double().permute(0, 3, 1, 2), 7, padding=3, stride=2)  # [n, 3 * 49, p * q]
    ref = torch.einsum("npk,ncp->kc", dy.cpu().double().reshape(n, p * q, 64), cols).reshape(64, 3, 7, 7)
    assert ref.abs().max() < 2048
    assert torch.equal(dw.cpu().double(), ref.permute(0, 2, 3, 1))
