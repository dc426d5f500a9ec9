"""Rounding error of the FP32 Wilson kernel on smooth links, against FP64 of the same FP32 inputs: no
larger than 5.65e-8 of the norm, what a sum of three complex products per component gives (a root mean
square over 8 million numbers: it moves by a thousandth between fields). The order of the chains of
multiply-adds decides it: in the order of the columns they give 5.70e-8."""
import numpy as np
import pytest

import synth
from oracle import wilson
from tests.gpu_util import ctx, rel, M0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1, 2])
def test_f32_rounding_error(variant):
    dims = (8, 16, 16, 16)
    U = synth.gauge_links(dims, 0.3, 1001)
    v = synth.gaussian_source(dims, 302).astype(np.complex64)
    c = ctx(dims, U, a=0.1, b=2.6, wilson_variant=variant)
    out = np.zeros_like(v)
    c.wilson_apply(v, out, 1)
    c.close()
    err = rel(out.astype(np.complex128), wilson.apply_K(U, v.astype(np.complex128), M0, False))
    print("variant %d: %.3e" % (variant, err))
    assert err <= 5.65e-8
