"""The FP32 sign of a context with kernel low-mode deflation (FP64 eigenvectors, FP32 solution)
against the spectral sign. Bound: the sign's stopping accuracy eta and as much again for
FP32 rounding (which the sign itself keeps below eta at 1e-5)."""
import numpy as np
import pytest

import synth
from oracle import wilson
from tests.gpu_util import ctx, rel, M0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [0, 1])
@pytest.mark.parametrize("n", [1, 5])
def test_f32_sign_with_kernel_deflation(method, n):
    dims, eta = (4, 4, 4, 4), 1e-5
    U = synth.gauge_links(dims, 0.3, 1001)
    w, Q = np.linalg.eigh(wilson.dense_K(U, M0))
    S = (Q * np.sign(w)) @ np.conj(Q.T)
    c = ctx(dims, U, a=0.95 * np.abs(w).min(), b=1.05 * np.abs(w).max(), n_poles=20, eps=1e-8, sign_method=method)
    c.kernel_deflate(6, tol=1e-11, max_iter=200)
    v = synth.gaussian_source(dims, 2101, nvec=n).reshape((n,) + tuple(reversed(dims)) + (4, 3))
    out = np.zeros_like(v)
    c.sign_apply(v, out, eta=eta, prec=1)
    c.close()
    for j in range(n):
        assert rel(out[j].ravel(), S @ v[j].ravel()) <= 2 * eta
