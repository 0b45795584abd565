"""What a user of the library has it do, as cases that can be timed and compared.

Every case goes through the public entry points (paper_1911_07384_gb300.pf16 and
the ResNet50 training step over it), over the range from a single small
convolution (N = 4) to the whole batch-256 training step:

  conv    one convolution layer: forward, data gradient, weight gradient
  block   a bottleneck residual block with identity shortcut, forward and
          backward, in the training step's call sequence (fused statistics,
          shortcut gradient added in the data gradient)
  stem    the network's stem: 7x7 convolution, BatchNorm + ReLU + max pooling,
          and their backward
  bn      a BatchNorm layer on its own, forward and backward
  head    average pooling, classifier, softmax cross-entropy and their backward
  update  the gradient average over the ranks (this rank's share) and the SGD
          step over the parameters
  step    a whole ResNet-50 training step, captured once in a CUDA graph

All tensors are binary16; the library takes any 2-byte dtype, so they are
torch.float16 here.
"""
from __future__ import annotations

import math

import torch

from paper_1911_07384_gb300 import pf16
from paper_1911_07384_gb300.resnet50 import LR, MOMENTUM, WD, ResNet50

F16 = torch.float16
ONE, QUARTER = 0x3C00, 0x3400  # binary16 bits of the BatchNorm output scales 1 and 0.25


def _value(bits):
    return torch.tensor([bits], dtype=torch.int16).view(F16).double().item()


EPS = _value(0x00A8)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest calls: one 64-channel 3x3 layer at batch 4, where launches
        # and latency are the time
        {"name": "conv 3x3 56 64-64 n4", "kind": "conv", "n": 4, "h": 56, "w": 56, "c": 64, "k": 64, "r": 3,
         "stride": 1, "f32": False},
        # the most frequent 3x3 of ResNet-50 (stage 3) at the sweep's batch 64
        {"name": "conv 3x3 14 256-256 n64", "kind": "conv", "n": 64, "h": 14, "w": 14, "c": 256, "k": 256, "r": 3,
         "stride": 1, "f32": False},
        # a strided 3x3 (the first block of stage 2): the data gradient has stride phases
        {"name": "conv 3x3s2 56 128-128 n64", "kind": "conv", "n": 64, "h": 56, "w": 56, "c": 128, "k": 128, "r": 3,
         "stride": 2, "f32": False},
        # pure-GEMM 1x1 layers at batch 256: balanced between tensor cores and
        # memory, and bound by memory
        {"name": "conv 1x1 14 1024-256 n256", "kind": "conv", "n": 256, "h": 14, "w": 14, "c": 1024, "k": 256, "r": 1,
         "stride": 1, "f32": False},
        {"name": "conv 1x1 56 256-64 n256", "kind": "conv", "n": 256, "h": 56, "w": 56, "c": 256, "k": 64, "r": 1,
         "stride": 1, "f32": False},
        # odd sizes, channels that fill no tile, the FP32-accumulation option
        {"name": "conv 3x3 27 192-320 n13 f32", "kind": "conv", "n": 13, "h": 27, "w": 27, "c": 192, "k": 320, "r": 3,
         "stride": 1, "f32": True},
        # an identity block of stage 2, forward and backward
        {"name": "block 28 512-128 n64", "kind": "block", "n": 64, "h": 28, "c": 512, "width": 128},
        # the stem at half the headline batch
        {"name": "stem 224 n128", "kind": "stem", "n": 128, "image": 224},
        # a block's last BatchNorm (residual, ReLU) on its own
        {"name": "bn 28 512 n64 residual", "kind": "bn", "n": 64, "h": 28, "w": 28, "c": 512, "residual": True},
        # the network's head at the headline batch
        {"name": "head 7 2048-1000 n256", "kind": "head", "n": 256, "hw": 49, "c": 2048, "classes": 1000},
        # all of ResNet-50's decayed parameters, averaged over 8 ranks
        {"name": "update 25.5M world 8", "kind": "update", "params": 25503912, "world": 8},
        # the headline: one training step at batch 256
        {"name": "step n256 224", "kind": "step", "n": 256, "image": 224},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# no drawn layer holds more activations, or costs more operations, than these
_MOST_PIXELS_CHANNELS = 256 * 56 * 56 * 256
_MOST_FLOPS = 60e9


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "conv", "block", "stem", "bn", "head", "update", "step"])
    if kind == "conv":
        while True:
            r = rng.choice([1, 3])
            stride = rng.choice([1, 1, 2])
            n, h = _log_int(rng, 1, 256), _log_int(rng, 7, 56)
            w = h if rng.random() < 0.7 else _log_int(rng, 7, 56)
            c, k = 64 * _log_int(rng, 1, 32), 64 * _log_int(rng, 1, 32)
            case = {"kind": "conv", "n": n, "h": h, "w": w, "c": c, "k": k, "r": r, "stride": stride,
                    "f32": rng.random() < 0.15}
            if n * h * w * max(c, k) <= _MOST_PIXELS_CHANNELS and 1e8 < work(case)["flops"] / 3 < _MOST_FLOPS:
                return case
    if kind == "block":
        while True:
            width = 64 * _log_int(rng, 1, 8)
            case = {"kind": "block", "n": _log_int(rng, 2, 256), "h": _log_int(rng, 7, 56), "c": 4 * width,
                    "width": width}
            if case["n"] * case["h"] ** 2 * case["c"] <= _MOST_PIXELS_CHANNELS // 2 and \
                    1e8 < work(case)["flops"] / 3 < _MOST_FLOPS:
                return case
    if kind == "stem":
        return {"kind": "stem", "n": _log_int(rng, 2, 256), "image": 32 * rng.randint(2, 7)}
    if kind == "bn":
        while True:
            case = {"kind": "bn", "n": _log_int(rng, 1, 256), "h": _log_int(rng, 5, 112), "w": _log_int(rng, 5, 112),
                    "c": 8 * _log_int(rng, 1, 256), "residual": rng.random() < 0.5}
            if case["n"] * case["h"] * case["w"] * case["c"] <= _MOST_PIXELS_CHANNELS // 2:
                return case
    if kind == "head":
        return {"kind": "head", "n": _log_int(rng, 4, 512), "hw": rng.choice([9, 16, 25, 36, 49, 64]),
                "c": 64 * _log_int(rng, 8, 32), "classes": 8 * _log_int(rng, 2, 256)}
    if kind == "update":
        return {"kind": "update", "params": 8 * _log_int(rng, 36864 // 8, 25503912 // 8), "world": _log_int(rng, 1, 128)}
    return {"kind": "step", "n": _log_int(rng, 8, 224), "image": 32 * rng.randint(3, 7)}


# -------------------------------------------------------------------- helpers
def _normal(gen, shape, std=1.0, mean=0.0):
    return torch.empty(shape, device="cuda", dtype=torch.float32).normal_(mean, std, generator=gen).to(F16)


def _uninit(*shape):
    return torch.empty(shape, device="cuda", dtype=F16)


def _bytes(n):
    return torch.empty(max(int(n), 256), device="cuda", dtype=torch.uint8)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _weights(gen, k, r, c):  # KRSC, He-normal
    return _normal(gen, (k, r, r, c), math.sqrt(2.0 / (r * r * c)))


def _out(h, r, stride):
    return (h + 2 * (r // 2) - r) // stride + 1


def _desc(n, h, w, c, k, r, stride=1):
    return pf16.conv_desc(n, h, w, c, k, r, r, stride, r // 2)


class _Norm:
    """A BatchNorm's parameters, saved statistics, gradients and ReLU mask, as a program keeps them."""

    def __init__(self, gen, n, h, w, c, scale=QUARTER, relu=True, residual=False):
        flags = (pf16.PF16_BN_RELU if relu else 0) | (pf16.PF16_BN_RESIDUAL if residual else 0)
        self.desc = pf16.bn_desc(n, h, w, c, 0x00A8, scale, flags)
        self.gamma, self.beta = _normal(gen, (c,), 0.1, 1.0), _normal(gen, (c,), 0.1)
        self.mean, self.invstd, self.dgamma, self.dbeta = (_uninit(c) for _ in range(4))
        self.mask = _bytes(n * h * w * c // 8) if relu else None
        self.ws_bytes = pf16.bn_workspace_size(self.desc)

    def fwd(self, ws, x, y, residual=None, stats=None):
        pf16.bn_fwd_bwd(self.desc, 0, ws, x=x, gamma=self.gamma, beta=self.beta, residual=residual, y=y,
                        mean=self.mean, invstd=self.invstd, relu_mask=self.mask, conv_stats=stats)

    def bwd(self, ws, x, dy, dx, dresidual=None, stats=None):
        pf16.bn_fwd_bwd(self.desc, 1, ws, x=x, gamma=self.gamma, mean=self.mean, invstd=self.invstd, dy=dy,
                        relu_mask=self.mask, dx=dx, dgamma=self.dgamma, dbeta=self.dbeta, dresidual=dresidual,
                        conv_stats=stats)


# ----------------------------------------------------------------------- conv
def _conv_inputs(case, seed):
    g = _gen(seed)
    n, h, w, c, k, r, st = (case[f] for f in ("n", "h", "w", "c", "k", "r", "stride"))
    x = _normal(g, (n, h, w, c))
    wt = _weights(g, k, r, c)
    dy = _normal(g, (n, _out(h, r, st), _out(w, r, st), k), 0.01)
    return x, wt, dy


def _prepare_conv(case, seed):
    x, wt, dy = _conv_inputs(case, seed)
    d = _desc(case["n"], case["h"], case["w"], case["c"], case["k"], case["r"], case["stride"])
    ws = _bytes(max(pf16.conv_workspace_size(d, p) for p in
                    (pf16.PF16_PASS_FWD, pf16.PF16_PASS_DGRAD, pf16.PF16_PASS_WGRAD)))
    return {"kind": "conv", "d": d, "x": x, "w": wt, "dy": dy, "y": torch.empty_like(dy), "dx": torch.empty_like(x),
            "dw": torch.empty_like(wt), "ws": ws, "flags": pf16.PF16_F32_ACCUM if case["f32"] else 0}


def _run_conv(s):
    pf16.conv_fwd(s["d"], s["x"], s["w"], s["y"], s["ws"], s["flags"])
    pf16.conv_dgrad(s["d"], s["dy"], s["w"], s["dx"], s["ws"], s["flags"])
    pf16.conv_wgrad(s["d"], s["x"], s["dy"], s["dw"], s["ws"], s["flags"])
    return {"y": s["y"], "dx": s["dx"], "dw": s["dw"]}


def _nchw(t):
    return t.permute(0, 3, 1, 2)


def _nhwc(t):
    return t.permute(0, 2, 3, 1).contiguous()


def _conv64(x, wt, stride=1):
    """y of an NHWC binary64 input and KRSC weights: a sum over the filter taps, each a matrix product."""
    n, h, w, c = x.shape
    k, r = wt.shape[0], wt.shape[1]
    p, q = _out(h, r, stride), _out(w, r, stride)
    pad = torch.nn.functional.pad(x, (0, 0, r // 2, r // 2, r // 2, r // 2))
    y = torch.zeros(n * p * q, k, dtype=torch.float64, device=x.device)
    for a in range(r):
        for b in range(r):
            rows = pad[:, a:a + (p - 1) * stride + 1:stride, b:b + (q - 1) * stride + 1:stride, :]
            y += rows.reshape(n * p * q, c) @ wt[:, a, b, :].t()
    return y.reshape(n, p, q, k)


def _conv64_dx(dy, wt, h, w, stride=1):
    n, p, q, k = dy.shape
    r, c = wt.shape[1], wt.shape[3]
    pad = torch.zeros(n, h + 2 * (r // 2) + stride, w + 2 * (r // 2) + stride, c, dtype=torch.float64, device=dy.device)
    for a in range(r):
        for b in range(r):
            pad[:, a:a + (p - 1) * stride + 1:stride, b:b + (q - 1) * stride + 1:stride, :] += \
                (dy.reshape(n * p * q, k) @ wt[:, a, b, :]).reshape(n, p, q, c)
    return pad[:, r // 2:r // 2 + h, r // 2:r // 2 + w, :].contiguous()


def _conv64_dw(x, dy, r, stride=1):
    n, p, q, k = dy.shape
    c = x.shape[3]
    pad = torch.nn.functional.pad(x, (0, 0, r // 2, r // 2, r // 2, r // 2))
    dw = torch.empty(k, r, r, c, dtype=torch.float64, device=x.device)
    for a in range(r):
        for b in range(r):
            rows = pad[:, a:a + (p - 1) * stride + 1:stride, b:b + (q - 1) * stride + 1:stride, :]
            dw[:, a, b, :] = dy.reshape(n * p * q, k).t() @ rows.reshape(n * p * q, c)
    return dw


def _exact_conv(case, seed):
    x, wt, dy = (t.double() for t in _conv_inputs(case, seed))
    st = case["stride"]
    return {"y": _conv64(x, wt, st), "dx": _conv64_dx(dy, wt, case["h"], case["w"], st),
            "dw": _conv64_dw(x, dy, case["r"], st)}


def _work_conv(case):
    n, h, w, c, k, r, st = (case[f] for f in ("n", "h", "w", "c", "k", "r", "stride"))
    px, po = n * h * w, n * _out(h, r, st) * _out(w, r, st)
    nx, ny, nw = px * c, po * k, k * r * r * c
    return {"bytes": 2.0 * (2 * nx + 2 * ny + 2 * nw), "flops": 3 * 2.0 * po * k * c * r * r}


# ---------------------------------------------------------------------- block
def _block_inputs(case, seed):
    g = _gen(seed)
    n, h, c, wd = case["n"], case["h"], case["c"], case["width"]
    t = {"x_prev": _normal(g, (n, h, h, c)),  # the last conv's output of the block before
         "shift": _normal(g, (n, h, h, c), 0.5),  # that block's shortcut
         "dy": _normal(g, (n, h, h, c), 0.01),
         "w1": _weights(g, wd, 1, c), "w2": _weights(g, wd, 3, wd), "w3": _weights(g, c, 1, wd)}
    norms = [_Norm(g, n, h, h, c, residual=True), _Norm(g, n, h, h, wd), _Norm(g, n, h, h, wd),
             _Norm(g, n, h, h, c, residual=True)]  # the block before's last, and this block's three
    return t, norms


def _prepare_block(case, seed):
    n, h, c, wd = case["n"], case["h"], case["c"], case["width"]
    t, norms = _block_inputs(case, seed)
    d = [_desc(n, h, h, c, wd, 1), _desc(n, h, h, wd, wd, 3), _desc(n, h, h, wd, c, 1)]
    wide = {k: _uninit(n, h, h, c) for k in ("x", "a3", "y", "da3", "dx", "da_prev")}
    thin = {k: _uninit(n, h, h, wd) for k in ("a1", "b1", "a2", "b2", "db2", "da2", "db1", "da1")}
    dw = {"dw%d" % i: torch.empty_like(t["w%d" % i]) for i in (1, 2, 3)}
    ws = _bytes(max([pf16.conv_workspace_size(x, pf16.PF16_PASS_WGRAD) for x in d] + [m.ws_bytes for m in norms]))
    s = {"kind": "block", "d": d, "norms": norms, "ws": ws, **t, **wide, **thin, **dw}
    s["fstats"] = [_bytes(pf16.conv_bnstats_size(x)) for x in d]
    s["bstats"] = [_bytes(pf16.conv_dgrad_bnstats_size(x)) for x in d]
    # the block before's last BatchNorm: its output is this block's input
    norms[0].fwd(ws, s["x_prev"], s["x"], residual=s["shift"])
    return s


def _run_block(s):
    (d1, d2, d3), (prev, n1, n2, n3), ws, f, b = s["d"], s["norms"], s["ws"], s["fstats"], s["bstats"]
    pf16.conv_fwd_bnstats(d1, s["x"], s["w1"], s["a1"], f[0])
    n1.fwd(ws, s["a1"], s["b1"], stats=f[0])
    pf16.conv_fwd_bnstats(d2, s["b1"], s["w2"], s["a2"], f[1])
    n2.fwd(ws, s["a2"], s["b2"], stats=f[1])
    pf16.conv_fwd_bnstats(d3, s["b2"], s["w3"], s["a3"], f[2])
    n3.fwd(ws, s["a3"], s["y"], residual=s["x"], stats=f[2])
    n3.bwd(ws, s["a3"], s["dy"], s["da3"])
    pf16.conv_wgrad(d3, s["b2"], s["da3"], s["dw3"], ws)
    pf16.conv_dgrad_bnstats(d3, s["da3"], s["w3"], s["db2"], s["a2"], n2.mask, n2.mean, n2.invstd, b[2])
    n2.bwd(ws, s["a2"], s["db2"], s["da2"], stats=b[2])
    pf16.conv_wgrad(d2, s["b1"], s["da2"], s["dw2"], ws)
    pf16.conv_dgrad_bnstats(d2, s["da2"], s["w2"], s["db1"], s["a1"], n1.mask, n1.mean, n1.invstd, b[1])
    n1.bwd(ws, s["a1"], s["db1"], s["da1"], stats=b[1])
    pf16.conv_wgrad(d1, s["x"], s["da1"], s["dw1"], ws)
    pf16.conv_dgrad_bnstats_add(d1, s["da1"], s["w1"], s["dx"], s["x_prev"], prev.mask, prev.mean, prev.invstd,
                                s["dy"], n3.mask, b[0])
    prev.bwd(ws, s["x_prev"], s["dx"], s["da_prev"], stats=b[0])
    out = {k: s[k] for k in ("y", "dx", "da_prev", "dw1", "dw2", "dw3")}
    for i, m in enumerate((prev, n1, n2, n3)):
        out["dgamma%d" % i], out["dbeta%d" % i] = m.dgamma, m.dbeta
    return out


class _Norm64:
    """A BatchNorm (biased variance, output times the scale, optional residual and ReLU) in binary64."""

    def __init__(self, m, x, residual=None, relu=True):
        self.s, self.gamma, self.relu = _value(m.desc.post_scale), m.gamma.double(), relu
        c = x.shape[-1]
        flat = x.reshape(-1, c)
        self.mean, var = flat.mean(0), flat.var(0, unbiased=False)
        self.invstd = 1.0 / (var + EPS).sqrt()
        self.xhat = (x - self.mean) * self.invstd
        y = (self.xhat * self.gamma + m.beta.double()) * self.s
        self.y = y if residual is None else y + residual
        if relu:
            self.y = self.y.relu()

    def bwd(self, dy):
        """(dx, dgamma, dbeta, the gradient where the ReLU passed)"""
        if self.relu:
            dy = dy * (self.y > 0)
        c = dy.shape[-1]
        a, b = dy.reshape(-1, c), self.xhat.reshape(-1, c)
        m1, m2 = a.mean(0), (a * b).mean(0)
        dx = self.s * self.gamma * self.invstd * (dy - m1 - self.xhat * m2)
        return dx, self.s * (a * b).sum(0), self.s * a.sum(0), dy


def _exact_block(case, seed):
    if _work_block(case)["flops"] > 300e9:
        return None
    t, (mp, m1, m2, m3) = _block_inputs(case, seed)
    t = {k: v.double() for k, v in t.items()}
    prev = _Norm64(mp, t["x_prev"], t["shift"])
    x = prev.y
    h = case["h"]
    n1 = _Norm64(m1, _conv64(x, t["w1"]))
    n2 = _Norm64(m2, _conv64(n1.y, t["w2"]))
    n3 = _Norm64(m3, _conv64(n2.y, t["w3"]), x)
    out = {"y": n3.y}
    da3, out["dgamma3"], out["dbeta3"], dsc = n3.bwd(t["dy"])
    out["dw3"] = _conv64_dw(n2.y, da3, 1)
    da2, out["dgamma2"], out["dbeta2"], _ = n2.bwd(_conv64_dx(da3, t["w3"], h, h))
    out["dw2"] = _conv64_dw(n1.y, da2, 3)
    da1, out["dgamma1"], out["dbeta1"], _ = n1.bwd(_conv64_dx(da2, t["w2"], h, h))
    out["dw1"] = _conv64_dw(x, da1, 1)
    out["dx"] = _conv64_dx(da1, t["w1"], h, h) + dsc
    out["da_prev"], out["dgamma0"], out["dbeta0"], _ = prev.bwd(out["dx"])
    return out


def _work_block(case):
    px, c, wd = case["n"] * case["h"] ** 2, case["c"], case["width"]
    nw = 2 * c * wd + 9 * wd * wd
    # in: x, dy, the BatchNorm input before; out: y, dx, its gradient
    return {"bytes": 2.0 * (6 * px * c + 2 * nw), "flops": 3 * 2.0 * px * nw}


# ----------------------------------------------------------------------- stem
def _stem_inputs(case, seed):
    g = _gen(seed)
    n, im = case["n"], case["image"]
    h = _out(im, 7, 2)
    p = _out(h, 3, 2)
    x, wt = _normal(g, (n, im, im, 3)), _weights(g, 64, 7, 3)
    return x, wt, _Norm(g, n, h, h, 64, ONE), _normal(g, (n, p, p, 64), 0.01)


def _prepare_stem(case, seed):
    x, wt, norm, dp = _stem_inputs(case, seed)
    n, h, p = case["n"], norm.desc.h, dp.shape[1]
    d = _desc(n, case["image"], case["image"], 3, 64, 7, 2)
    ws = _bytes(max(pf16.conv_workspace_size(d, pf16.PF16_PASS_FWD), pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD),
                    norm.ws_bytes))
    return {"kind": "stem", "n": n, "h": h, "d": d, "x": x, "w": wt, "norm": norm, "dp": dp, "ws": ws,
            "a": _uninit(n, h, h, 64), "p": torch.empty_like(dp), "arg": _bytes(n * p * p * 64),
            "stats": _bytes(pf16.conv_bnstats_size(d)), "db": _uninit(n, h, h, 64), "da": _uninit(n, h, h, 64),
            "dw": torch.empty_like(wt)}


def _run_stem(s):
    m, ws = s["norm"], s["ws"]
    pf16.conv_fwd_bnstats(s["d"], s["x"], s["w"], s["a"], s["stats"], ws)
    pf16.bn_relu_maxpool_fwd(m.desc, ws, s["p"], s["arg"], x=s["a"], gamma=m.gamma, beta=m.beta, mean=m.mean,
                             invstd=m.invstd, relu_mask=m.mask, conv_stats=s["stats"])
    pf16.maxpool_bwd_argmax(s["arg"], s["dp"], s["db"], s["n"], s["h"], s["h"], 64)
    m.bwd(ws, s["a"], s["db"], s["da"])
    pf16.conv_wgrad(s["d"], s["x"], s["da"], s["dw"], ws)
    return {"a": s["a"], "p": s["p"], "da": s["da"], "dw": s["dw"], "dgamma": m.dgamma, "dbeta": m.dbeta}


def _exact_stem(case, seed):
    x, wt, m, _ = _stem_inputs(case, seed)
    a = _conv64(x.double(), wt.double(), 2)
    norm = _Norm64(m, a)
    p = torch.nn.functional.max_pool2d(_nchw(norm.y), 3, 2, 1)
    # the backward follows the positions of the maxima, which rounding decides where values tie
    return {"a": a, "p": _nhwc(p), "da": None, "dw": None, "dgamma": None, "dbeta": None}


def _work_stem(case):
    n, im = case["n"], case["image"]
    h = _out(im, 7, 2)
    p = _out(h, 3, 2)
    na, np_ = n * h * h * 64, n * p * p * 64
    return {"bytes": 2.0 * (2 * n * im * im * 3 + 3 * na + 2 * np_), "flops": 2 * 2.0 * na * 147}


# ------------------------------------------------------------------------- bn
def _bn_inputs(case, seed):
    g = _gen(seed)
    n, h, w, c = (case[f] for f in ("n", "h", "w", "c"))
    x = (_normal(g, (n, h, w, c)).float() * (0.5 + torch.rand(c, device="cuda", generator=g)) +
         torch.randn(c, device="cuda", generator=g)).to(F16)
    res = _normal(g, (n, h, w, c)) if case["residual"] else None
    return x, res, _normal(g, (n, h, w, c), 0.01), _Norm(g, n, h, w, c, residual=case["residual"])


def _prepare_bn(case, seed):
    x, res, dy, m = _bn_inputs(case, seed)
    return {"kind": "bn", "x": x, "res": res, "dy": dy, "norm": m, "y": torch.empty_like(x), "dx": torch.empty_like(x),
            "dres": torch.empty_like(x) if res is not None else None, "ws": _bytes(m.ws_bytes)}


def _run_bn(s):
    m = s["norm"]
    m.fwd(s["ws"], s["x"], s["y"], residual=s["res"])
    m.bwd(s["ws"], s["x"], s["dy"], s["dx"], dresidual=s["dres"])
    return {"y": s["y"], "mean": m.mean, "invstd": m.invstd, "dx": s["dx"], "dres": s["dres"], "dgamma": m.dgamma,
            "dbeta": m.dbeta}


def _exact_bn(case, seed):
    x, res, dy, m = _bn_inputs(case, seed)
    n = _Norm64(m, x.double(), res.double() if res is not None else None)
    dx, dg, db, dr = n.bwd(dy.double())
    return {"y": n.y, "mean": n.mean, "invstd": n.invstd, "dx": dx, "dres": dr if res is not None else None,
            "dgamma": dg, "dbeta": db}


def _work_bn(case):
    e = case["n"] * case["h"] * case["w"] * case["c"]
    # forward x, y (and the residual); backward x, dy, dx (and its gradient); the ReLU bits both ways
    return {"bytes": 2.0 * e * (7 if case["residual"] else 5) + e / 4, "flops": 0.0}


# ----------------------------------------------------------------------- head
def _head_inputs(case, seed):
    g = _gen(seed)
    n, hw, c, k = (case[f] for f in ("n", "hw", "c", "classes"))
    x = _normal(g, (n, hw, c)).relu()
    w, bias = _normal(g, (k, c), math.sqrt(2.0 / c)), _normal(g, (k,), 0.01)
    return x, w, bias, torch.randint(0, k, (n,), device="cuda", generator=g, dtype=torch.int32)


def _prepare_head(case, seed):
    n, hw, c, k = (case[f] for f in ("n", "hw", "c", "classes"))
    x, w, bias, labels = _head_inputs(case, seed)
    d = _desc(n, 1, 1, c, k, 1)
    ws = _bytes(max(pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD), pf16.softmax_xent_workspace_size(n, k)))
    return {"kind": "head", "n": n, "hw": hw, "c": c, "k": k, "d": d, "x": x, "w": w, "bias": bias, "labels": labels,
            "ws": ws, "f": _uninit(n, c), "logits": _uninit(n, k), "loss": _uninit(8)[:1], "dlogits": _uninit(n, k),
            "dbias": torch.empty_like(bias), "dw": torch.empty_like(w), "df": _uninit(n, c), "dx": torch.empty_like(x)}


def _run_head(s):
    n, hw, c, k = s["n"], s["hw"], s["c"], s["k"]
    pf16.avgpool_fwd(s["x"], s["f"], n, hw, c)
    pf16.conv_fwd(s["d"], s["f"], s["w"], s["logits"])
    pf16.softmax_xent(s["logits"], s["bias"], s["labels"], n, k, s["loss"], s["dlogits"], s["dbias"], s["ws"])
    pf16.conv_wgrad(s["d"], s["f"], s["dlogits"], s["dw"], s["ws"])
    pf16.conv_dgrad(s["d"], s["dlogits"], s["w"], s["df"])
    pf16.avgpool_bwd(s["df"], s["dx"], n, hw, c)
    return {key: s[key] for key in ("f", "logits", "loss", "dlogits", "dbias", "dw", "df", "dx")}


def _exact_head(case, seed):
    x, w, bias, labels = _head_inputs(case, seed)
    n, hw, k = case["n"], case["hw"], case["classes"]
    f = x.double().mean(1)
    logits = f @ w.double().t()
    z = logits + bias.double()
    lab = labels.long()
    loss = torch.nn.functional.cross_entropy(z, lab).reshape(1)
    dl = (z.softmax(1) - torch.nn.functional.one_hot(lab, k)) / n
    df = dl @ w.double()
    return {"f": f, "logits": logits, "loss": loss, "dlogits": dl, "dbias": dl.sum(0), "dw": dl.t() @ f, "df": df,
            "dx": (df / hw).unsqueeze(1).expand(-1, hw, -1).contiguous()}


def _work_head(case):
    n, hw, c, k = (case[f] for f in ("n", "hw", "c", "classes"))
    return {"bytes": 2.0 * (2 * n * hw * c + 2 * n * c + 2 * n * k + 2 * k * c), "flops": 3 * 2.0 * n * c * k}


# --------------------------------------------------------------------- update
def _update_inputs(case, seed):
    g = _gen(seed)
    n, world = case["params"], case["world"]
    share = -(-n // (8 * world)) * 8  # this rank's slice of the gradient, whole 16-byte pieces
    planes = _normal(g, (world, share), 0.01) if world > 1 else None
    return _normal(g, (n,), 0.05), _normal(g, (n,), 0.02), _normal(g, (n,), 0.01), planes


def _scale_bits(world):
    return torch.tensor([1.0 / world], dtype=torch.float64).to(F16).view(torch.int16).item()


def _prepare_update(case, seed):
    w, v, g, planes = _update_inputs(case, seed)
    return {"kind": "update", "w": w, "v": v, "g": g, "planes": planes, "world": case["world"],
            "scale": _scale_bits(case["world"]), "mean": _uninit(planes.shape[1]) if planes is not None else None}


def _run_update(s):
    out = {"w": s["w"], "v": s["v"]}
    if s["planes"] is not None:
        share = s["planes"].shape[1]
        pf16.allreduce_combine(s["planes"], s["world"], share, share, s["scale"], s["mean"])
        out["mean"] = s["mean"]
    pf16.sgd_update(s["w"], s["v"], s["g"], LR, MOMENTUM, WD)
    return out


def _exact_update(case, seed):
    w, v, g, planes = _update_inputs(case, seed)
    v = _value(MOMENTUM) * v.double() + g.double() + _value(WD) * w.double()
    out = {"w": w.double() - _value(LR) * v, "v": v}
    if planes is not None:
        out["mean"] = planes.double().sum(0) * _value(_scale_bits(case["world"]))
    return out


def _work_update(case):
    n, world = case["params"], case["world"]
    share = -(-n // (8 * world)) * 8
    return {"bytes": 10.0 * n + (2.0 * share * (world + 1) if world > 1 else 0.0), "flops": 0.0}


# ----------------------------------------------------------------------- step
def _prepare_step(case, seed):
    n, im = case["n"], case["image"]
    net = ResNet50(batch=n, image=im, seed_cfg=seed, wgrad_branch=True)
    g = _gen(seed)
    net.x.copy_(_normal(g, (n * im * im * 3,)).view(torch.int16))
    net.labels.copy_(torch.randint(0, net.classes, (n,), device="cuda", generator=g, dtype=torch.int32))
    # the residual branches take part, as they do after the first steps from the
    # zero-gamma initialisation
    for b in net.blocks:
        b.bn3.gamma.copy_(_normal(g, (b.bn3.c,), 0.05, 0.25).view(torch.int16))
    for a in (net.wd, net.nowd):
        for which in ("w", "v"):
            a.__dict__["start_" + which] = getattr(a, which).clone()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        net.step()  # an eager step first: one-time set-up stays outside the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        net.step()
    for a in (net.wd, net.nowd):
        for which in ("w", "v"):
            getattr(a, which).copy_(a.__dict__.pop("start_" + which))
    torch.cuda.synchronize()
    return {"kind": "step", "net": net, "graph": graph}


def _run_step(s):
    s["graph"].replay()
    net = s["net"]
    return {"loss": net.loss.view(F16), "logits": net.logits.view(F16), "w": net.wd.w.view(F16),
            "bn": net.nowd.w.view(F16)}


def _work_step(case):
    """The convolutions' operations, and each layer boundary's tensors once: activations
    written and read in the forward and read again in the backward, their gradients
    written and read."""
    from paper_1911_07384_gb300.resnet50 import conv_shapes

    flops, elems, weights = 0.0, 0, 0
    for i, (name, (n, h, w, c, k, r, s, st, pad)) in enumerate(conv_shapes(case["n"], case["image"])):
        p, q = (h + 2 * pad - r) // st + 1, (w + 2 * pad - s) // st + 1
        flops += 2.0 * n * p * q * k * c * r * s * (2 if i == 0 else 3)
        elems += n * p * q * k
        weights += k * r * s * c
    return {"bytes": 2.0 * 5 * elems + 10.0 * weights, "flops": flops}


# ------------------------------------------------------------------ interface
_PREPARE = {"conv": _prepare_conv, "block": _prepare_block, "stem": _prepare_stem, "bn": _prepare_bn,
            "head": _prepare_head, "update": _prepare_update, "step": _prepare_step}
_RUN = {"conv": _run_conv, "block": _run_block, "stem": _run_stem, "bn": _run_bn, "head": _run_head,
        "update": _run_update, "step": _run_step}
_WORK = {"conv": _work_conv, "block": _work_block, "stem": _work_stem, "bn": _work_bn, "head": _work_head,
         "update": _work_update, "step": _work_step}
_EXACT = {"conv": _exact_conv, "block": _exact_block, "stem": _exact_stem, "bn": _exact_bn, "head": _exact_head,
          "update": _exact_update}


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["kind"]](state)


def work(case):
    return _WORK[case["kind"]](case)


def exact(case, seed):
    fn = _EXACT.get(case["kind"])
    return fn(case, seed) if fn else None


def tolerance(case):
    """About four times what the same call shows with its sums in another order."""
    kind = case["kind"]
    if kind == "update":
        return "exact"  # every operation and its order are given
    if kind == "conv":
        if case["f32"]:  # one rounding of each result; the weight gradient's partial sums are binary16
            return {"rel": 0.002, "max": 0.02}
        # binary16 accumulation over the filter's taps and channels, and over at
        # least 4,096 pixels in the weight gradient: 6.3e-4 measured at 576 terms,
        # 1.7e-3 at 2,304, 4.8e-3 at 18,432, 2.2e-3 for weight gradients
        terms = case["r"] ** 2 * max(case["c"], case["k"])
        rel = min(0.03, 4 * (3e-4 + 4e-5 * math.sqrt(max(terms, 4096))))
        return {"rel": rel, "max": min(0.9, 9 * rel)}
    if kind == "head":
        return {"rel": 0.02, "max": 0.2}
    if kind == "step":  # logits 3.7e-3 to 5.2e-3, weights 2.5e-4 (largest 2e-2)
        return {"rel": 0.02, "max": 0.1}
    # BatchNorm and ReLU: a value near zero that rounds to the other side turns its
    # gradient on or off (block 6e-2, stem 9e-3, with the statistics in another order)
    return {"rel": 0.03, "max": 0.99}
