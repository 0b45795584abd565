"""The BatchNorm's finals at the edges of their trees: one to 304 statistics CTAs
(chunks of 256 rows at 8 and 24 channels), powers of two and their neighbours,
ragged last chunks and several chunks per CTA.  test_finals_tree replays the
finals' trees in binary16 from the per-CTA results that the statistics kernels
leave in the workspace, with row counts taken from the chunk layout: equal bits.
test_finals checks the whole pass against binary64, within the bounds of the
BatchNorm itself (wide enough to hide a slot): the mean within (L + 2) u max|x|,
invstd within (2 L + 8) u, the backward sums within (4 L + 8) u sum|terms|, L =
ceil(log2 R), u = 2^-11."""
import numpy as np
import pytest

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300 import synthetic as syn
from gpu_util import U, dev, empty16, f64, host, workspace

pytestmark = pytest.mark.gpu

EPS = float(np.uint16(0x00A8).view(np.float16))


ROWS = [1, 7, 256, 257, 31 * 256 + 5, 33 * 256, 152 * 256 + 1, 255 * 256 + 1, 257 * 256 - 3,
        303 * 256 + 7, 700 * 256 + 3]


def _inputs(R, C):
    x = (f64(syn.normal_f16(61, (R, C))) * 2 + np.linspace(-1, 1, C)).astype(np.float16).view(np.uint16)
    return x, syn.normal_f16(62, (R, C), 0.01)


@pytest.mark.parametrize("R", ROWS)
@pytest.mark.parametrize("C", [8, 24])
def test_finals(R, C):
    L = int(np.ceil(np.log2(max(R, 2))))
    x, dy = _inputs(R, C)
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


def _rn(v):  # binary16, roundTiesToEven (of exact binary64 sums and products of two binary16 numbers)
    return np.asarray(v, np.float64).astype(np.float16).astype(np.float64)


def _merge(a, b):
    """Two (mean, variance, rows) nodes by the count-aware pairwise rule, one rounding per operation."""
    (am, av, an), (bm, bv, bn) = a, b
    if an == 0 or bn == 0:
        return a if bn == 0 else b
    halves = lambda p, q: _rn(p / 2 + _rn(q / 2))
    d = _rn(bm - am)
    if an == bn:
        dh = _rn(d / 2)
        return halves(am, bm), _rn(halves(av, bv) + _rn(dh * dh)), an + bn
    wa, wb = (_rn(np.float32(k) / np.float32(an + bn)) for k in (an, bn))
    m = _rn(_rn(am * wa) + _rn(bm * wb))
    return m, _rn(_rn(_rn(av * wa) + _rn(bv * wb)) + _rn(_rn(d * d) * _rn(wa * wb))), an + bn


def _tree(nodes, empty, merge):
    """A slot per thread, two neighbours where there are more than 256; then threads t and t + half."""
    if len(nodes) > 256:
        nodes = nodes + [empty] * (len(nodes) % 2)
        nodes = [merge(nodes[i], nodes[i + 1]) for i in range(0, len(nodes), 2)]
    n = 1
    while n < len(nodes):
        n *= 2
    nodes = nodes + [empty] * (n - len(nodes))
    while len(nodes) > 1:
        half = len(nodes) // 2
        nodes = [merge(nodes[i], nodes[i + half]) for i in range(half)]
    return nodes[0]


@pytest.mark.parametrize("R", ROWS)
@pytest.mark.parametrize("C", [8, 24])
def test_finals_tree(R, C):
    x, dy = _inputs(R, C)
    d = pf16.bn_desc(1, 1, R, C, 0x00A8, 0x3400, 0)  # outputs times 1/4
    ws = workspace(pf16.bn_workspace_size(d))
    tx, tg, tm, ti = dev(x), dev(np.full(C, 0x3C00, np.uint16)), empty16(C), empty16(C)
    chunks = [min(256, R - r) for r in range(0, R, 256)]
    slots = lambda n: ws.cpu().numpy()[:4 * n * C].view(np.float16).astype(np.float64).reshape(2, n, C)

    pf16.bn_fwd_bwd(d, 0, ws, x=tx, mean=tm, invstd=ti)  # statistics alone
    assert pf16.sync_status() == 0
    n = min(len(chunks), 304)  # CTA b has chunks b, b + n, ...
    means, variances = slots(n)
    mean, var, rows = _tree([(means[b], variances[b], sum(chunks[b::n])) for b in range(n)],
                            (np.zeros(C), np.zeros(C), 0), _merge)
    assert rows == R
    assert np.array_equal(f64(host(tm)), mean)
    ve = _rn(var + EPS)
    assert np.all(np.abs(f64(host(ti)) * np.sqrt(ve) - 1) <= 2 * U)  # one rounded reciprocal square root

    dx, dg, db = empty16(R * C), empty16(C), empty16(C)
    pf16.bn_fwd_bwd(d, 1, ws, x=tx, gamma=tg, mean=tm, invstd=ti, dy=dev(dy), dx=dx, dgamma=dg, dbeta=db)
    assert pf16.sync_status() == 0
    n = min(len(chunks), 152)
    for sums, out in zip(slots(n), (db, dg)):
        total = _tree(list(sums), np.zeros(C), lambda p, q: _rn(p + q))
        assert np.array_equal(f64(host(out)), _rn(total * 0.25))
