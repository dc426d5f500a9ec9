"""The waits between the blocks of a one-launch Lanczos cycle when their time runs out: the cycle is
done again by launches per step, in the first cycle as in later ones. Either result is within its
stopping bound of the same rational, so they differ by at most twice that. A short limit may let the
time run out anywhere."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,eta", [(1, 1e-5), (3, 1e-9)])
@pytest.mark.parametrize("cap", [0, 11])
def test_a_cycle_that_gave_up_is_done_again(prec, eta, cap):
    dims, n = (6, 2, 4, 6), 3
    U = synth.gauge_links(dims, 0.3, 81)
    v = synth.gaussian_source(dims, 83, nvec=n)
    v[1] = 0.0
    outs = []
    for limit in (2.0, 0.0):
        c = ctx(dims, U, n_poles=20, a=0.1, b=2.7, lanczos_cap=cap)
        c.set_wait_limit(limit)
        o = np.full_like(v, 7.0)
        c.sign_apply(v, o, eta=eta, prec=prec)
        one, stepped, _, _ = c.lanczos_cycles()
        assert (one > 0 and stepped == 0) if limit else (one == 0 and stepped > 0)
        outs.append(o)
        c.close()
    assert np.all(outs[1][1] == 0.0)
    for j in (0, 2):
        assert rel(outs[0][j], outs[1][j]) <= 2 * eta


@pytest.mark.parametrize("prec,eta", [(1, 1e-5), (3, 1e-9)])
def test_a_short_limit(prec, eta):
    dims, n = (8, 8, 8, 8), 2
    U = synth.gauge_links(dims, 0.3, 81)
    v = synth.gaussian_source(dims, 84, nvec=n)
    c = ctx(dims, U, n_poles=20, a=0.1, b=2.7, lanczos_cap=24)
    want = np.zeros_like(v)
    c.sign_apply(v, want, eta=eta, prec=prec)
    for limit in (1e-9, 1e-6, 1e-5, 1e-4):
        c.set_wait_limit(limit)
        o = np.zeros_like(v)
        c.sign_apply(v, o, eta=eta, prec=prec)
        for j in range(n):
            assert rel(o[j], want[j]) <= 2 * eta, limit
    c.close()
