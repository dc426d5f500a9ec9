"""K in FP32 straight into the caller's single-precision device buffer."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import ctx, rel

pytestmark = pytest.mark.gpu

# K is a sum of 8 x 6 products per component: two FP32 evaluations of it differ by a few roundings of
# the largest terms, 2^-24 sqrt(100) of the norm at most
K_TOL = 6e-7


@pytest.mark.parametrize("dims,n", [((2, 2, 2, 2), 1), ((10, 6, 14, 12), 3), ((10, 6, 6, 2), 7), ((8, 8, 8, 8), 2)])
def test_wilson_into_the_callers_buffer(dims, n):
    """Single-precision device buffers: aligned, a view off a 16-byte boundary, and in place."""
    U = synth.gauge_links(dims, 0.3, 95)
    c = ctx(dims, U, a=0.1, b=2.6, wilson_variant=0)
    psi = synth.gaussian_source(dims, 96, nvec=n).astype(np.complex64)
    ref = np.zeros_like(psi)
    c.wilson_apply(psi, ref, 1)            # host buffers: K and the unpacking apart
    d = torch.from_numpy(psi).cuda()
    out = torch.full_like(d, 7.0)
    c.wilson_apply(d, out, prec=1)
    big = torch.full((d.numel() + 2,), 7.0, dtype=d.dtype, device="cuda")
    c.wilson_apply(d, big[1:-1].view(d.shape), prec=1)
    c.wilson_apply(d, d, prec=1)
    for got in (out, big[1:-1].view(d.shape), d):
        for j in range(n):
            assert rel(got.cpu().numpy()[j], ref[j]) <= K_TOL
    assert big[0] == 7.0 and big[-1] == 7.0
