"""The weight gradient's split-K plan, through the workspace it asks for: the
split count minimising the makespan model over every count from 1 to 1,024."""
import random

from paper_1911_07384_gb300 import pf16


def _cdiv(a, b):
    return -(-a // b)


def _splits(pixels, k, ncols):
    bn = 256 if ncols % 256 == 0 else 192 if ncols % 192 == 0 else 128 if ncols % 128 == 0 else \
        64 if ncols <= 64 else 192 if ncols <= 192 else 256
    tiles, num_kb = _cdiv(k, 128) * _cdiv(ncols, bn), _cdiv(pixels, 64)
    t_kb, dw = 0.4e-6 * bn / 256.0, 2.0 * k * ncols
    best, splits = -1.0, _cdiv(num_kb, min(num_kb, 64))
    for sp in range(1, 1025):
        kps = _cdiv(num_kb, sp)
        if kps > 64:
            continue
        if kps < 4 and sp > 1:
            break
        real = _cdiv(num_kb, kps)
        t = _cdiv(tiles * real, 152) * (kps * t_kb + 1.0e-6) + (real * dw * 2.0 / 2e12 if real > 1 else 0.0)
        if best < 0 or t < best * (1 - 1e-9):
            best, splits = t, real
    return splits if splits <= 1024 else _cdiv(num_kb, _cdiv(num_kb, 1024))


def test_split_counts():
    rng = random.Random(7)
    shapes = [(1, 1, 1, 64, 64), (2, 7, 7, 64, 64), (1, 16, 16, 64, 64), (1, 15, 17, 64, 64), (256, 14, 14, 1024, 256),
              (256, 128, 128, 64, 64), (300, 130, 130, 128, 64)]
    shapes += [(rng.randint(1, 256), rng.randint(1, 60), rng.randint(1, 60), 64 * rng.randint(1, 32),
                64 * rng.randint(1, 32)) for _ in range(300)]
    for n, h, w, c, k in shapes:
        d = pf16.conv_desc(n, h, w, c, k, 1, 1, 1, 0)
        sp = _splits(n * h * w, k, c)
        want = 0 if sp == 1 else (sp * k * c * 2 + 255) // 256 * 256
        assert pf16.conv_workspace_size(d, pf16.PF16_PASS_WGRAD) == want, (n, h, w, c, k)
