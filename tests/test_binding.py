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


def test_current_stream_without_the_private_functions(monkeypatch):
    """The current stream comes through torch's public call where the two private ones are missing."""
    torch = pytest.importorskip("torch")

    class Stream:
        cuda_stream = 0x5150

    monkeypatch.setattr(pf16, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: Stream())
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    assert pf16._stream(None) == 0x5150
    assert pf16._stream(7) == 7 and pf16._stream(Stream()) == 0x5150
