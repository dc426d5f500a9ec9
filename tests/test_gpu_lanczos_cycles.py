"""Systems of one batch that finish in different cycles of the stored-basis Lanczos: eigenvectors of K
(two steps at most) beside vectors that fill several cycles, against the exact sign. What a finished
system added to its solution must stay as it is in the cycles that the others still need."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx, dense_4444, rel

pytestmark = pytest.mark.gpu


# two systems: the one-launch form where the precision has one; six: launches per step
@pytest.mark.parametrize("prec,eta", [(0, 1e-9), (1, 1e-5), (3, 1e-9)])
@pytest.mark.parametrize("n", [2, 6])
def test_systems_that_finish_in_earlier_cycles(prec, eta, n):
    U, Kd, S, w = dense_4444()
    Q = np.linalg.eigh(Kd)[1]
    dims = (4, 4, 4, 4)
    c = ctx(dims, U, n_poles=20, eps=1e-10, a=0.95 * np.abs(w).min(), b=1.05 * np.abs(w).max(), lanczos_cap=11)
    v = synth.gaussian_source(dims, 301, nvec=n)
    v[1] = (Q[:, 40] * 3.0).reshape(v[1].shape)
    v[n - 1] = (Q[:, 7] + 1j * Q[:, -9]).reshape(v[1].shape)
    out = np.zeros_like(v)
    c.sign_apply(v, out, eta=eta, prec=prec)
    c.close()
    for j in range(n):
        # the stopping accuracy, and as much for rounding and the rational's bound
        assert rel(out[j].ravel(), S @ v[j].ravel()) <= 2 * eta, j
