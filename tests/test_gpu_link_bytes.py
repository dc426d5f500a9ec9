"""Algorithmic bytes of a Wilson launch are the same everywhere: what the profiler books for a sign of
known steps is made of the spinors and links that bench_wilson counts, links once per launch."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,cls,spinor,link", [(0, "wilson_f64", 192, 384), (1, "wilson_f32", 96, 192),
                                                  (3, "wilson_f64e", 192, 576)])
def test_link_bytes_are_the_same_everywhere(prec, cls, spinor, link):
    dims, n, steps = (4, 4, 4, 4), 5, 6
    V = 256
    c = ctx(dims, synth.gauge_links(dims, 0.3, 81), n_poles=20, a=0.1, b=2.7, wilson_variant=0, mscg_max=steps)
    assert c.bench_wilson(prec, n, 2)[1] == V * (2 * spinor * n + link)
    v = synth.gaussian_source(dims, 84, nvec=n)
    c.profile_reset()
    c.profile_enable(True)
    with pytest.raises(lib().OvlError):           # the iteration limit: exactly `steps` steps per system
        c.sign_apply(v, np.zeros_like(v), eta=1e-5, prec=prec)
    c.profile_enable(False)
    b = c.profile_get()[cls]["bytes"]
    # per step K reads W and writes t, L reads t, W_j and (after the first) W_{j-1} and writes W_{j+1}; the
    # final application reads y, v and writes the result (FP64)
    lanczos = n * steps * 4 * spinor + n * (2 * steps - 1) * spinor + 2 * steps * link
    final = n * (spinor + 2 * 192) + link
    assert b == V * (lanczos + final)
    c.close()
