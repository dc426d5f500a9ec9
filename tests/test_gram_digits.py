"""A host model of the FP32-arithmetic digit splitting of the tensor-core Gram blocks for FP64
operands: digits in the ranges that the exact FP32 accumulation needs (128, then 64), and the
element reconstructed to the truncation (2^-47) plus the last digit's rounding (2^-43)."""
import math
from fractions import Fraction

import numpy as np

F = np.float32
MAGIC = F(12582912.0)


def fma(a, b, c):
    return F(np.float64(a) * np.float64(b) + np.float64(c))   # both operands have at most 24 bits


def split64(x, e):
    b = int(np.float64(x).view(np.uint64))
    lo, hi = b & 0xffffffff, b >> 32
    t, sg = (hi >> 20) & 0x7ff, hi & 0x80000000
    if t < max(e + 897, 1):
        return F(0), F(0)
    ex = t - 896 - e
    h = np.uint32((ex << 23) | ((b >> 29) & 0x7fffff) | sg).view(np.float32)
    scale = np.uint32(0 if ex <= 25 else ((ex - 25) << 23) | sg).view(np.float32)
    return h, F(F((lo >> 6) & 0x7fffff) * scale)


def digit(s, r):
    t = fma(s, F(128), MAGIC)
    return int(F(t - MAGIC)), fma(r, F(128), F(MAGIC - t))


def digits(x, e):
    r, low = split64(x, e)
    out = []
    for k in range(6):
        if k == 2:
            d, r = digit(fma(low, F(0.0078125), r), r)
            r = F(r + low)
        else:
            d, r = digit(r, r)
        out.append(d)
    return out


def test_fp32_digits_of_fp64_elements():
    rng = np.random.default_rng(1)
    edges = [1.0, 1 - 2.0 ** -53, 0.5, 1 - 2.0 ** -24, 1 - 2.0 ** -25, 127.5 / 128, 0.5 - 2.0 ** -40, -1 + 2.0 ** -30,
             2.0 ** -20, 2.0 ** -30 + 2.0 ** -60, 2.0 ** -43, 2.0 ** -44, 2.0 ** -60, 0.0, 63.5 / 128 - 2.0 ** -22,
             (63.5 + 63.5 / 128) / 128, 1 - 2.0 ** -21 - 2.0 ** -45]
    for scale in (2.0 ** -100, 1.0, 2.0 ** 58):
        v = np.concatenate([np.array(edges), rng.uniform(-1, 1, 3000),
                            rng.standard_normal(1000) * np.exp(-30 * rng.random(1000))]) * scale
        e = max(math.frexp(abs(x))[1] for x in v if x)
        for x in v:
            d = digits(x, e)
            assert abs(d[0]) <= 128 and all(abs(k) <= 64 for k in d[1:])
            val = sum(Fraction(k, 1 << (7 * (s + 1))) for s, k in enumerate(d))
            assert abs(val - Fraction(float(x)) / Fraction(2) ** e) <= Fraction(2) ** -43 * Fraction(9, 8)
