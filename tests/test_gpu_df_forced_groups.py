"""A forced number of double-float thread groups holds on any lattice (only the other precisions'
tiles need extents that divide): four groups (variant 2) on lattices whose pairs do not fill a block,
K against the oracle and a sign against FP64, both within their stopping bounds of one rational."""
import numpy as np
import pytest

import synth
from oracle import wilson
from tests.gpu_util import ctx, rel, M0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (10, 6, 2, 2), (6, 2, 4, 6)])
def test_forced_groups_on_ragged_lattices(dims):
    U = synth.gauge_links(dims, 0.3, 61)
    v = synth.gaussian_source(dims, 62, nvec=3)
    ref = [wilson.apply_K(U, x, M0, False) for x in v]
    want, out = np.zeros_like(v), np.zeros_like(v)
    for variant in range(4):
        c = ctx(dims, U, n_poles=20, a=0.1, b=2.7, wilson_variant=variant)
        assert [c.wilson_tuning(p)[0] for p in range(4)] == 3 * [variant if variant == 1 else 0] + [variant]
        c.wilson_apply(v, out, 3)
        for j in range(3):
            assert rel(out[j], ref[j]) <= 2e-13
        if variant == 0:
            c.sign_apply(v, want, eta=1e-10, prec=0)
        c.sign_apply(v, out, eta=1e-10, prec=3)
        c.close()
        for j in range(3):
            assert rel(out[j], want[j]) <= 2e-10
