"""The head's kernels at the edges of their splits, bit for bit: the average
pooling's halving tree over padded pixels (runs of one, several and many
batches per warp; one to eight sets of channel groups per CTA), and the loss's
column and loss trees over row segments.
The expected trees are numpy float16 arithmetic (correctly rounded adds;
a/2 + rn(b/2) formed exactly in binary64 and rounded once)."""
import numpy as np
import pytest
import torch

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300 import synthetic as syn
from gpu_util import dev, empty16, host, workspace

pytestmark = pytest.mark.gpu


def _half_merge(a, b):
    h = (b.astype(np.float64) / 2).astype(np.float16).astype(np.float64)
    return (a.astype(np.float64) / 2 + h).astype(np.float16)


def _halving_tree(v):  # over axis 0, zero padded to a power of two
    n = 1
    while n < v.shape[0]:
        n *= 2
    v = np.concatenate([v, np.zeros((n - v.shape[0],) + v.shape[1:], np.float16)])
    while v.shape[0] > 1:
        v = _half_merge(v[0::2], v[1::2])
    return v[0], n


def _f16(bits):
    return np.asarray(bits, np.uint16).view(np.float16)


@pytest.mark.parametrize("N,HW,C", [(3, 1, 8), (2, 2, 264), (5, 7, 64), (1, 8, 8), (2, 9, 40), (3, 33, 72), (2, 65, 8),
                                    (1, 2049, 8), (70, 3, 72), (50, 12, 40), (40, 20, 72), (300, 1, 8)])
def test_avgpool_tree(N, HW, C):
    x = syn.normal_f16(31, (N, HW, C))
    y, dx = empty16(N * C), empty16(N * HW * C)
    pf16.avgpool_fwd(dev(x), y, N, HW, C)
    mean, n2 = _halving_tree(_f16(x).transpose(1, 0, 2))
    want = mean * np.float16(n2 / HW)
    assert np.array_equal(_f16(host(y)).reshape(N, C), want)
    dy = syn.normal_f16(32, (N, C))
    pf16.avgpool_bwd(dev(dy), dx, N, HW, C)
    assert pf16.sync_status() == 0
    want = np.repeat((_f16(dy) * np.float16(1.0 / HW))[:, None, :], HW, 1)
    assert np.array_equal(_f16(host(dx)).reshape(N, HW, C), want)


@pytest.mark.parametrize("B,K,bias", [(1, 8, True), (2, 1, False), (33, 32, True), (40, 4096, True), (1023, 33, True),
                                      (1025, 7, False), (2100, 5, True)])
def test_softmax_trees(B, K, bias):
    logits = syn.normal_f16(33, (B, K), 2.0)
    b = dev(syn.normal_f16(34, (K,), 0.1)) if bias else None
    labels = torch.from_numpy(syn.labels(35, B, K)).cuda()
    loss, dl, db = empty16(1), empty16(B * K), empty16(K)
    ws = workspace(pf16.softmax_xent_workspace_size(B, K))
    pf16.softmax_xent(dev(logits), b, labels, B, K, loss, dl, db, ws)
    assert pf16.sync_status() == 0
    v = _f16(host(dl)).reshape(B, K)
    while v.shape[0] > 1:  # pairwise; a missing right node passes its left one through
        odd = v[-1:] if v.shape[0] % 2 else v[:0]
        v = np.concatenate([v[0:v.shape[0] - len(odd):2] + v[1::2], odd])
    assert np.array_equal(_f16(host(db)), v[0])
    rows = ws.cpu().numpy().view(np.uint16)[:B]
    mean, n2 = _halving_tree(_f16(rows))
    assert np.array_equal(_f16(host(loss))[0], mean * np.float16(n2 / B))
    loss2, dl2 = empty16(1), empty16(B * K)
    pf16.softmax_xent(dev(logits), b, labels, B, K, loss2, dl2, None, ws)  # no bias gradient
    assert np.array_equal(host(loss2), host(loss)) and np.array_equal(host(dl2), host(dl))
