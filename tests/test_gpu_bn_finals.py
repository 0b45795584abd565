"""The BatchNorm's finals at the edges of their trees: one to 304 statistics CTAs
(chunks of 256 rows at 8 channels), powers of two and their neighbours, ragged
last chunks and several chunks per CTA.  Bounds as for the BatchNorm itself: the
mean within (L + 2) u max|x|, invstd within (2 L + 8) u, the backward sums
within (4 L + 8) u sum|terms|, L = ceil(log2 R), u = 2^-11."""
import numpy as np
import pytest

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300 import synthetic as syn
from gpu_util import U, dev, empty16, f64, host, workspace

pytestmark = pytest.mark.gpu

EPS = float(np.uint16(0x00A8).view(np.float16))


@pytest.mark.parametrize("R", [1, 7, 256, 257, 31 * 256 + 5, 33 * 256, 152 * 256 + 1, 255 * 256 + 1, 257 * 256 - 3,
                               303 * 256 + 7, 700 * 256 + 3])
@pytest.mark.parametrize("C", [8, 24])
def test_finals(R, C):
    L = int(np.ceil(np.log2(max(R, 2))))
    x = (f64(syn.normal_f16(61, (R, C))) * 2 + np.linspace(-1, 1, C)).astype(np.float16).view(np.uint16)
    dy = syn.normal_f16(62, (R, C), 0.01)
    gamma, beta = np.full(C, 0x3C00, np.uint16), np.zeros(C, np.uint16)
    d = pf16.bn_desc(1, 1, R, C, 0x00A8, 0x3C00, 0)
    ws = workspace(pf16.bn_workspace_size(d))
    tx, tg, y, tm, ti = dev(x), dev(gamma), empty16(R * C), empty16(C), empty16(C)
    pf16.bn_fwd_bwd(d, 0, ws, x=tx, gamma=tg, beta=dev(beta), y=y, mean=tm, invstd=ti)
    dx, dg, db = empty16(R * C), empty16(C), empty16(C)
    pf16.bn_fwd_bwd(d, 1, ws, x=tx, gamma=tg, mean=tm, invstd=ti, dy=dev(dy), dx=dx, dgamma=dg, dbeta=db)
    assert pf16.sync_status() == 0
    v = f64(x).reshape(R, C)
    mean, invstd = v.mean(0), 1 / np.sqrt(v.var(0) + EPS)
    assert np.all(np.abs(f64(host(tm)) - mean) <= (L + 2) * U * np.abs(v).max(0))
    if R > 8:  # (a handful of rows: the variance's own rounding is relative to max|x|^2)
        assert np.all(np.abs(f64(host(ti)) - invstd) <= (2 * L + 8) * U * invstd)
    g = f64(dy).reshape(R, C)
    xhat = (v - f64(host(tm))) * f64(host(ti))  # the kernels' own saved statistics
    tol = (4 * L + 8) * U
    assert np.all(np.abs(f64(host(db)) - g.sum(0)) <= tol * np.abs(g).sum(0) + 2.0 ** -24)
    assert np.all(np.abs(f64(host(dg)) - (g * xhat).sum(0)) <= tol * (np.abs(g) * (np.abs(xhat) + 1)).sum(0) + 2.0 ** -24)
