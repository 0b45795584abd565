"""The Python binding's marshalling, as far as it goes without a GPU."""
import pytest

from paper_1911_07384_gb300 import pf16


class _Tensor:
    """What the binding asks of a tensor."""

    nbytes = 1 << 20

    def data_ptr(self):
        return 4096


def test_batchnorm_ignores_other_keywords():
    """A keyword that names no BatchNorm tensor is ignored, as by the structure's own
    constructor: the call gets as far as the library's check of the workspace."""
    d = pf16.bn_desc(1, 4, 4, 8, 0x00A8, 0x3C00, 0)
    tensors = {k: _Tensor() for k in ("x", "gamma", "beta", "y", "mean", "invstd")}
    with pytest.raises(pf16.PF16Error, match="workspace"):
        pf16.bn_fwd_bwd(d, 0, None, stream=0, momentum=_Tensor(), name=None, **tensors)
    del tensors["y"]
    d = pf16.bn_desc(1, 4, 4, 8, 0x00A8, 0x3C00, pf16.PF16_BN_RELU)
    with pytest.raises(pf16.PF16Error, match="workspace"):
        pf16.bn_relu_maxpool_fwd(d, None, _Tensor(), _Tensor(), stream=0, momentum=_Tensor(), **tensors)
