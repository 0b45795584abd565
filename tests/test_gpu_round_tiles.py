"""The 128-wide tiles of launches whose last round of 256-wide ones would leave
SMs idle: an image's outputs do not depend on the tile width, so the first images
of a batch that takes the narrow tiles come out bit for bit as in a smaller batch
that takes the wide ones.  And the two epilogues of the backward statistics on
either side of their line (four and five K-blocks, several tiles per CTA)."""
import pytest

import test_gpu_convbn as convbn
import test_gpu_tile_fill as fill

pytestmark = pytest.mark.gpu

# h, w, c, k, r, stride; images in the 256-wide and in the 128-wide launch
CASES = [(7, 7, 512, 512, 1, 1, 150, 256), (7, 7, 512, 512, 3, 1, 150, 256), (28, 28, 320, 320, 1, 1, 12, 64),
         (14, 14, 512, 128, 3, 2, 40, 64), (13, 15, 256, 256, 3, 1, 98, 110)]


@pytest.mark.parametrize("h,w,c,k,r,st,small,large", CASES)
def test_same_bits(h, w, c, k, r, st, small, large):
    fill.test_tile_width(h, w, c, k, r, st, small, large)


# dx channels and dy channels: 3, 4, 5 and 8 K-blocks, one and several N tiles, 192- and 320-wide rows
STATS = [(48, 28, 256, 192), (48, 28, 256, 256), (48, 28, 256, 320), (29, 28, 320, 320), (40, 28, 192, 512)]


@pytest.mark.parametrize("n,h,c,k", STATS)
def test_backward_statistics(orc, n, h, c, k):
    convbn.test_conv_dgrad_bnstats_then_bn_bwd(orc, ((n, h, h, c, k, 1, 1, 1, 0), True))
