"""The pipelined BatchNorm + ReLU + max pooling where its CTAs walk several tiles
and the ring of stages wraps: bit for bit the separate calls, at the stem's own
size, at odd sizes (partial last tiles, images of one tile), with two stages, and
on either side of the rule that chooses it."""
import pytest

from paper_1911_07384_gb300 import pf16
from gpu_util import dev, workspace
from test_gpu_stem_fused import EPS, bn_inputs, fused_fwd, separate_fwd

import torch

pytestmark = pytest.mark.gpu

# tiles (two output rows): 896, 1,200, 609, 700 (one per image), 936 (rows of 128 x 64: two stages); then one tile
# in all, the widest rows of two stages, and what the pipeline leaves out: one stage, five channel groups
SHAPES = [(16, 112, 112, 64), (150, 31, 30, 64), (21, 113, 45, 128), (700, 3, 40, 16), (26, 143, 128, 64),
          (1, 1, 1, 8), (3, 21, 176, 64), (3, 21, 177, 64), (5, 33, 30, 40)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "N{}_{}x{}_C{}".format(*s))
def test_pipeline(shape):
    N, H, W, C = shape
    d = pf16.bn_desc(N, H, W, C, EPS, 0x3C00, pf16.PF16_BN_RELU)
    ws = workspace(pf16.bn_workspace_size(d))
    x, gamma, beta = bn_inputs(shape, 71)
    args = (d, ws, dev(x), dev(gamma), dev(beta), None, N, H, W, C)
    for a, b in zip(separate_fwd(*args), fused_fwd(*args)):
        assert torch.equal(a, b)
