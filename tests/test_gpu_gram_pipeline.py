"""Lengths of the Gram kernel's pipeline at which its chunks and buffers can go wrong: a range
shorter than its three buffers or a chunk, one stage past a chunk (84 stages in five splits: 16
and 17), whole chunks, and every operand type, against NumPy in FP64. Bound: each operand is
represented to 9/8 2^-43 of at most twice its vector's largest element."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,na,nb", [((14, 2, 2, 2), 330, 300), ((2, 2, 2, 2), 1, 3), ((4, 4, 2, 2), 65, 130),
                                        ((8, 8, 2, 2), 64, 64)])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("g5", [0, 1])
def test_gram_pipeline_lengths(dims, na, nb, prec, g5):
    c = ctx(dims, synth.unit_links(dims), a=0.2, b=2.6)
    rng = np.random.default_rng(7)
    shp = tuple(reversed(dims)) + (4, 3)
    dt = np.complex128 if prec == 0 else np.complex64
    A = (rng.standard_normal((na,) + shp) + 1j * rng.standard_normal((na,) + shp)).astype(dt)
    B = (rng.standard_normal((nb,) + shp) + 1j * rng.standard_normal((nb,) + shp)).astype(dt)
    A[0] *= 2.0 ** 40
    B[-1] *= 2.0 ** -30
    G = c.gram(A, B, g5=g5, prec=prec)
    A2, B2 = A.reshape(na, -1).astype(np.complex128), B.astype(np.complex128)
    if g5:
        B2[..., 2:, :] *= -1
    B2 = B2.reshape(nb, -1)
    amax = np.abs(A2.view(np.float64)).max(axis=1)[:, None]
    bmax = np.abs(B2.view(np.float64)).max(axis=1)[None, :]
    unit = 2 * 9 / 8 * 2.0 ** -43
    # every product off by the two representation errors (complex: two products per part), plus FP64 rounding
    k = A2.shape[1]
    bound = 2 * 2 * k * unit * amax * bmax * 2
    assert np.all(np.abs(G - np.conj(A2) @ B2.T) <= bound)
    scale = np.linalg.norm(A2, axis=1)[:, None] * np.linalg.norm(B2, axis=1)[None, :]
    assert np.max(np.abs(G - np.conj(A2) @ B2.T) / scale) <= 1e-12


def test_pack_from_an_unaligned_view():
    """A device tensor that starts 8 bytes into an allocation takes the element-wise form."""
    import torch
    dims = (6, 2, 4, 6)
    V = 6 * 2 * 4 * 6
    c = ctx(dims, synth.gauge_links(dims, 0.3, 71), a=0.1, b=2.7)
    for prec in (1, 3):
        x = torch.from_numpy(synth.gaussian_source(dims, 72, nvec=2).astype(np.complex64)).cuda()
        big = torch.zeros(x.numel() + 2, dtype=torch.complex64, device="cuda")
        view = big[1:1 + x.numel()].view(x.shape)
        view.copy_(x)
        o1, big2 = torch.empty_like(x), torch.zeros_like(big)
        o2 = big2[1:1 + x.numel()].view(x.shape)
        c.wilson_apply(x, o1, prec)
        c.wilson_apply(view, o2, prec)
        assert view.data_ptr() % 16 == 8 and torch.equal(o1, o2)
        assert big2[0] == 0 and big2[-1] == 0
