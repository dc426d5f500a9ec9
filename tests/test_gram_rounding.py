"""FP64 operands of the tensor-core Gram blocks are rounded, not cut, to their six digits: a host
model of the splitting (leading 24 bits, the other 29 rounded to 24, digits by FP32 arithmetic) over
many elements at once. Elements on the grid are exact, an element is off by at most 9/8 2^-43 of its vector's scale, by the mean of a rounding (no bias; cutting
gives 2^-47), digits stay in the ranges of the exact FP32 sums. On the GPU: diagonal entries of
Gaussian vectors have no common offset."""
import numpy as np
import pytest

import synth

F = np.float32
MAGIC, C128 = F(12582912.0), F(128)


def fma(a, b, c):
    return (a.astype(np.float64) * np.float64(b) + np.asarray(c, dtype=np.float64)).astype(F)


def split64(x, e):
    b = x.view(np.uint64)
    lo, hi = b & np.uint64(0xffffffff), b >> np.uint64(32)
    t, sg = ((hi >> np.uint64(20)) & np.uint64(0x7ff)).astype(np.int64), (hi & np.uint64(0x80000000)).astype(np.uint32)
    zero = t < max(e + 897, 1)
    ex = np.where(zero, 1, t - 896 - e)
    h = ((ex << 23).astype(np.uint32) | ((b >> np.uint64(29)) & np.uint64(0x7fffff)).astype(np.uint32) | sg).view(F)
    v = (lo & np.uint64(0x1fffffff)).astype(F)
    scale = np.where(ex <= 31, np.uint32(0), (np.maximum(ex - 31, 0) << 23).astype(np.uint32) | sg).view(F)
    return np.where(zero, F(0), h), np.where(zero, F(0), v * scale)


def digits(x, e):
    r, low = split64(x, e)
    out = []
    for k in range(6):
        s = fma(low, F(0.0078125), r) if k == 2 else r
        t = fma(s, C128, MAGIC)
        out.append((t - MAGIC).astype(np.int64))
        r = fma(r, C128, MAGIC - t)
        if k == 2:
            r = r + low
    return out


def test_elements_are_rounded_without_bias():
    rng = np.random.default_rng(2)
    e = 0
    grid = rng.integers(-2 ** 42 + 1, 2 ** 42, 200000).astype(np.float64) / 2.0 ** 42
    gauss = rng.standard_normal(400000)
    gauss = gauss[np.abs(gauss) < 4] / 4
    full = rng.uniform(-1, 1, 400000)
    for x, exact in ((grid, True), (gauss, False), (full, False)):
        d = digits(x, e)
        assert np.abs(d[0]).max() <= 128 and max(np.abs(k).max() for k in d[1:]) <= 64
        # x minus its digits, exact in FP64: the sum of the first four is within 2^-29 of x
        rest = x - sum(k * 2.0 ** (-7 * (s + 1)) for s, k in enumerate(d[:4]))
        err = rest - sum(k * 2.0 ** (-7 * (s + 5)) for s, k in enumerate(d[4:]))
        if exact:
            assert np.all(err == 0)
            continue
        assert np.abs(err).max() <= 9 / 8 * 2.0 ** -43
        # the signed error outwards: five sigma of a mean of roundings, uniform in +-2^-43
        sigma = 2.0 ** -43 / np.sqrt(3 * len(x))
        assert abs(np.mean(err * np.sign(x))) <= 5 * sigma < 2.0 ** -48


def test_group_sums_stay_exact_at_the_digit_bounds():
    """Digits up to 128, then 64: what 512 reals of a group can sum to is an exact FP32 integer."""
    most = [128] + 5 * [64]
    for g in range(7):
        assert 512 * sum(most[s] * most[g - s] for s in range(6) if 0 <= g - s < 6) <= 1 << 24


@pytest.mark.gpu
def test_diagonal_entries_have_no_common_offset():
    """64 Gaussian vectors of 196608 reals. An element's rounding, uniform in +-2^-43 of a scale of 8, is a
    relative 1.3e-15 of a diagonal entry, of the mean over 64 entries 1.6e-16; the double-float sums add
    about as much. Held to 2e-15; cut elements are off by 1e-14."""
    import torch
    from tests.gpu_util import ctx
    dims, n = (8, 8, 8, 16), 64
    c = ctx(dims, synth.unit_links(dims), a=0.2, b=2.6)
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    A = torch.randn((n,) + tuple(reversed(dims)) + (4, 3), generator=g, device="cuda", dtype=torch.complex128)
    G = c.gram(A, A)
    c.close()
    n2 = torch.view_as_real(A).flatten(1).square().sum(1).cpu().numpy()
    off = np.mean((np.diag(G).real - n2) / n2)
    print("mean offset of the diagonal %.2e" % off)
    assert abs(off) <= 2e-15
