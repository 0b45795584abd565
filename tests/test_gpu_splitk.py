"""The weight gradient's split-K reduction at its edges: the partial planes the
GEMM leaves in the workspace, summed by numpy as the reduction's float16 tree
over the splits (zero padded), must be dw bit for bit -- one to hundreds of
splits, runs of one split to 128, whole and partial CTAs, dense results and the
patch GEMM's padded columns."""
import numpy as np
import pytest
import torch

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300 import synthetic as syn
from gpu_util import dev, empty16, host, workspace

pytestmark = pytest.mark.gpu


def _tree(v, chunks):
    """The splits in aligned runs, a run summed neighbours first, the runs' sums at a
    stride; as many runs, up to 256, as give 152 x 512 threads at one per run and chunk."""
    n = 1
    while n < v.shape[0]:
        n *= 2
    v = np.concatenate([v, np.zeros((n - v.shape[0],) + v.shape[1:], np.float16)])
    runs = 1
    while runs < n and runs < 256 and chunks * runs < 152 * 512:
        runs *= 2
    while v.shape[0] > runs:
        v = v[0::2] + v[1::2]
    while v.shape[0] > 1:
        half = v.shape[0] // 2
        v = v[:half] + v[half:]
    return v[0]


# n, h, w, c, k, r: splits 2 to several hundred (1x1 and strided 3x3: planes of k x r*r*c)
CASES = [(1, 16, 32, 64, 64, 1, 1), (1, 28, 28, 64, 64, 1, 1), (2, 28, 28, 64, 128, 1, 1), (5, 28, 28, 192, 64, 1, 1),
         (16, 56, 56, 64, 64, 1, 1), (40, 56, 56, 64, 64, 1, 1), (3, 31, 33, 64, 320, 3, 2)]


@pytest.mark.parametrize("n,h,w,c,k,r,st", CASES)
def test_tree_over_splits(n, h, w, c, k, r, st):
    p, q = (h + 2 * (r // 2) - r) // st + 1, (w + 2 * (r // 2) - r) // st + 1
    d = pf16.conv_desc(n, h, w, c, k, r, r, st, r // 2)
    x, dy = dev(syn.normal_f16(51, (n, h, w, c))), dev(syn.normal_f16(52, (n, p, q, k), 0.01))
    size = pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD)
    dw, ws, numel = empty16(k * r * r * c), workspace(size), k * r * r * c
    pf16.conv_wgrad(d, x, dy, dw, ws)
    assert pf16.sync_status() == 0
    splits = size // (2 * numel)
    assert splits > 1
    parts = ws.cpu().numpy()[:splits * numel * 2].view(np.float16).reshape(splits, numel)
    assert np.array_equal(host(dw), _tree(parts, numel // 8).view(np.uint16))


@pytest.mark.parametrize("n,h,c,k", [(256, 56, 256, 512), (84, 56, 1024, 1024)])
def test_long_runs(n, h, c, k):
    """Large results with many splits: runs of 32 and 128, which several threads share."""
    g = torch.Generator(device="cuda").manual_seed(57)
    f = lambda ch, std: torch.empty(n, h, h, ch, dtype=torch.float16, device="cuda").normal_(0.0, std, generator=g)
    d = pf16.conv_desc(n, h, h, c, k, 1, 1, 1, 0)
    size = pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD)
    dw, ws = empty16(k * c), workspace(size)
    pf16.conv_wgrad(d, f(c, 1.0), f(k, 0.01), dw, ws)
    assert pf16.sync_status() == 0
    splits = size // (2 * k * c)
    parts = ws.cpu().numpy()[:splits * k * c * 2].view(np.float16).reshape(splits, k * c)
    assert np.array_equal(host(dw), _tree(parts, k * c // 8).view(np.uint16))


def _padded_columns(x, dy, n, h, k):
    d = pf16.conv_desc(n, h, h, 3, k, 3, 3, 1, 1)
    size = pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD)
    dw, ws = empty16(k * 27), workspace(size)
    pf16.conv_wgrad(d, x, dy, dw, ws)
    assert pf16.sync_status() == 0
    patches = n * h * h * 32 * 2  # the patch matrix comes first in the workspace (a multiple of 256 bytes)
    splits = (size - patches) // (k * 32 * 2)
    parts = ws[patches:patches + splits * k * 64].cpu().numpy().view(np.float16).reshape(splits, k, 32)
    assert np.array_equal(host(dw).reshape(k, 27), _tree(parts, k * 4)[:, :27].view(np.uint16))
    return splits


def test_padded_columns():
    """A three-channel 3x3 convolution (patch GEMM): 27 columns of 32, the rest dropped."""
    n, h, k = 2, 24, 64
    _padded_columns(dev(syn.normal_f16(53, (n, h, h, 3))), dev(syn.normal_f16(54, (n, h, h, k), 0.01)), n, h, k)


def test_many_splits_of_a_small_result():
    """The same with 608 splits of 256 chunks: every thread of a CTA its own group."""
    n, h, k = 38, 224, 64
    g = torch.Generator(device="cuda").manual_seed(58)
    f = lambda ch, std: torch.empty(n, h, h, ch, dtype=torch.float16, device="cuda").normal_(0.0, std, generator=g)
    assert _padded_columns(f(3, 1.0), f(k, 0.01), n, h, k) > 512
