"""Cached graphs of sign iterations go when what they captured changes: the multi-shift form holds the
base shift sigma_0, which a kernel deflation moves while the pole count and every buffer stay the
same; and a batch that grows the Lanczos states moves them under the graphs of a smaller one."""
import numpy as np
import pytest

import synth
from oracle import wilson
from tests.gpu_util import ctx, rel, M0

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,eta", [(0, 1e-9), (3, 1e-9)])
def test_base_shift_of_a_new_rational(prec, eta):
    dims, npoles = (4, 4, 4, 4), 20
    U = synth.gauge_links(dims, 0.7, 1001)
    w, Q = np.linalg.eigh(wilson.dense_K(U, M0))
    S = (Q * np.sign(w)) @ np.conj(Q.T)
    c = ctx(dims, U, a=0.95 * np.abs(w).min(), b=1.05 * np.abs(w).max(), n_poles=npoles, eps=1e-9, sign_method=1)
    v = synth.gaussian_source(dims, 2201)
    exact = (S @ v.ravel()).reshape(v.shape)
    out = np.zeros_like(v)
    for n_ev in (None, 10, 0):
        if n_ev is not None:
            assert c.kernel_deflate(n_ev, tol=1e-11, max_iter=200, n_poles=npoles if n_ev else 0)[3] == npoles
        c.sign_apply(v, out, eta=eta, prec=prec)
        # the stopping accuracy, and the rational's own bound
        assert rel(out, exact) <= 2 * eta, n_ev
    c.close()


def test_states_that_grow_between_batches():
    dims, eta = (8, 8, 8, 8), 1e-5
    U = synth.gauge_links(dims, 0.3, 91)
    c = ctx(dims, U, n_poles=20, a=0.1, b=2.7)
    v = synth.gaussian_source(dims, 92, nvec=9)
    want, out = np.zeros_like(v), np.zeros_like(v)
    c.sign_apply(v, want, eta=1e-9, prec=3)
    d = ctx(dims, U, n_poles=20, a=0.1, b=2.7)
    for n in (5, 9, 5, 7, 5):
        o = np.zeros_like(v[:n])
        d.sign_apply(v[:n].copy(), o, eta=eta, prec=1)
        for j in range(n):
            assert rel(o[j], want[j]) <= 2 * eta
    c.close()
    d.close()
