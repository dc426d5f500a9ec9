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
