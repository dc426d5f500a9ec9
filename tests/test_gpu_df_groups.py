"""The double-float Wilson kernel keeps sites in pairs (i, i + V/2), in blocks of 32 pairs, and
shares the eight hops of a pair among 1, 2, 4 or 8 thread groups: every group count on
lattices whose pairs do not fill a block, with the shortest t (every hop in t changes halves)."""
import numpy as np
import pytest

import synth
from oracle import wilson
from tests.gpu_util import ctx, rel, M0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (10, 6, 2, 2), (6, 2, 4, 6), (4, 14, 2, 4)])
@pytest.mark.parametrize("apt", [0, 1])
def test_df_wilson_groups(dims, variant, apt):
    U = synth.gauge_links(dims, 0.3, 61)
    c = ctx(dims, U, a=0.1, b=2.6, bc_t=apt, wilson_variant=variant)
    psi = synth.gaussian_source(dims, 62, nvec=3)
    psi[1, 0, 0, 0, 0, 2, 1] *= 1e6        # a site far above the rest
    out = np.zeros_like(psi)
    c.wilson_apply(psi, out, 3)
    for j in range(3):
        assert rel(out[j], wilson.apply_K(U, psi[j], M0, bool(apt))) <= 2e-13


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 4, 6), (4, 14, 2, 4), (10, 6, 14, 12)])
@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("prec,eta,bound", [(3, 1e-10, 2e-10), (1, 1e-5, 2e-5)])
def test_sign_step_on_few_and_ragged_blocks(dims, n, prec, eta, bound):
    """The Lanczos step sums one partial per block of a launch: one to dozens of blocks, odd and
    even counts, small double-float blocks. Both signs are within their stopping bounds of the
    same rational, so they differ by at most the sum of the two."""
    U = synth.gauge_links(dims, 0.3, 63)
    c = ctx(dims, U, n_poles=20, a=0.1, b=2.7)
    v = synth.gaussian_source(dims, 64, nvec=n)
    ref, out = np.zeros_like(v), np.zeros_like(v)
    c.sign_apply(v, ref, eta=min(eta, 1e-10), prec=0)
    c.sign_apply(v, out, eta=eta, prec=prec)
    for j in range(n):
        assert rel(out[j], ref[j]) <= bound
