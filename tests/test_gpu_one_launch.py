"""The Lanczos iteration as one cooperative launch (small signs) against the launch-per-step form
(a forced launch shape): every tile shape it chooses by size, restarted cycles, systems of one
batch that stop at different steps, a zero vector, and the iteration limit. Both are within
their stopping bound of the same rational, so they differ by at most twice that."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx, lib, rel

pytestmark = pytest.mark.gpu


def _pair(dims, **kw):
    U = synth.gauge_links(dims, 0.3, 81)
    return [ctx(dims, U, n_poles=20, a=0.1, b=2.7, wilson_variant=v, **kw) for v in (-1, 0)]


# FP32: four warps per tile, one (up to 19 per SM), one (up to 27); double-float: 8 groups of 8
# pairs (up to 3 tiles per SM, 4), 2 groups of 16 (up to 5, 7); each size also past its neighbour's
@pytest.mark.parametrize("prec,dims,n", [(1, (4, 4, 4, 4), 1), (1, (8, 8, 8, 16), 4), (1, (16, 16, 16, 16), 1),
                                         (1, (16, 16, 16, 16), 2), (3, (2, 2, 2, 2), 4), (3, (8, 8, 8, 12), 1),
                                         (3, (8, 8, 8, 16), 1), (3, (8, 8, 8, 16), 2), (3, (8, 8, 8, 16), 4)])
def test_one_launch_matches_launch_per_step(prec, dims, n):
    eta = 1e-5 if prec == 1 else 1e-9
    v = synth.gaussian_source(dims, 82, nvec=n)
    outs = []
    for c in _pair(dims):
        o = np.zeros_like(v)
        c.sign_apply(v, o, eta=eta, prec=prec)
        outs.append(o)
        c.close()
    for j in range(n):
        assert rel(outs[0][j], outs[1][j]) <= 2 * eta


@pytest.mark.parametrize("prec", [1, 3])
def test_one_launch_restarts_and_uneven_systems(prec):
    dims = (6, 2, 4, 6)
    eta = 1e-5 if prec == 1 else 1e-9
    v = synth.gaussian_source(dims, 83, nvec=4)
    v[1] = 0.0
    v[2] = synth.point_source(dims, 1, 2)
    v[3] *= 1e-12
    outs = []
    for c in _pair(dims, lanczos_cap=11):
        o = np.full_like(v, 7.0)
        c.sign_apply(v, o, eta=eta, prec=prec)
        outs.append(o)
        c.close()
    assert np.all(outs[0][1] == 0.0)
    for j in (0, 2, 3):
        assert rel(outs[0][j], outs[1][j]) <= 2 * eta


@pytest.mark.parametrize("prec", [1, 3])
def test_one_launch_iteration_limit_is_reported(prec):
    B = lib()
    dims = (4, 4, 4, 4)
    c = ctx(dims, synth.gauge_links(dims, 0.3, 81), n_poles=20, a=0.1, b=2.7, mscg_max=9)
    v = synth.gaussian_source(dims, 84)
    with pytest.raises(B.OvlError) as e:
        c.sign_apply(v, np.zeros_like(v), eta=1e-6 if prec == 1 else 1e-9, prec=prec)
    assert e.value.status == B.OVL_ENOCONV
    o = np.zeros_like(v)
    c.sign_apply(v, o, eta=0.5, prec=prec)     # the context stays usable


@pytest.mark.parametrize("dims,n", [((10, 6, 14, 12), 1), ((6, 10, 14, 4), 4), ((10, 10, 10, 20), 1)])
def test_one_launch_four_groups(dims, n):
    """Double-float tiles of 8 pairs in four groups: up to 7 and up to 9 tiles per SM."""
    eta = 1e-9
    v = synth.gaussian_source(dims, 85, nvec=n)
    outs = []
    for c in _pair(dims):
        o = np.zeros_like(v)
        c.sign_apply(v, o, eta=eta, prec=3)
        outs.append(o)
        c.close()
    for j in range(n):
        assert rel(outs[0][j], outs[1][j]) <= 2 * eta
