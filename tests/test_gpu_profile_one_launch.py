"""The profiler describes what an unprofiled call runs: a small sign is one launch per Lanczos cycle
of its Wilson class and the final application, with the same result."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,cls,eta", [(1, "wilson_f32", 1e-5), (3, "wilson_f64e", 1e-9)])
@pytest.mark.parametrize("cap", [0, 16])
def test_profiled_sign_takes_the_same_form(prec, cls, eta, cap):
    dims = (4, 4, 4, 8)
    c = ctx(dims, synth.gauge_links(dims, 0.3, 81), n_poles=20, a=0.1, b=2.7, lanczos_cap=cap)
    v = synth.gaussian_source(dims, 83, nvec=2)
    plain, prof = np.zeros_like(v), np.zeros_like(v)
    c.sign_apply(v, plain, eta=eta, prec=prec)
    one = c.lanczos_cycles()[0]
    c.profile_reset()
    c.profile_enable(True)
    c.sign_apply(v, prof, eta=eta, prec=prec)
    c.profile_enable(False)
    cycles = c.lanczos_cycles()[0] - one
    r = c.profile_get()[cls]
    assert np.array_equal(plain, prof)
    assert cycles == (one if cap else 1) and c.lanczos_cycles()[1] == 0
    assert r["launches"] == cycles + 1 and r["ms"] > 0 and r["bytes"] > 0 and r["units"] > 0
    c.close()
