"""Which form a Lanczos cycle took (lanczos_cycles): the one-launch shapes that sizes choose, with a
forced launch shape none; and contexts in two threads whose launches of one kernel differ in size."""
import threading

import numpy as np
import pytest

import synth
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu
SMS = 152


def _tiles(dims, n, pairs, per_sm):
    V = int(np.prod(dims))
    tiles = (V // 2 + pairs - 1) // pairs * n if pairs else (V + 31) // 32 * n
    return tiles, -(-tiles // per_sm)


# precision, lattice, systems, groups, pairs of a tile (0: 32 sites)
@pytest.mark.parametrize("prec,dims,n,groups,pairs", [
    (1, (4, 4, 4, 4), 1, 4, 0), (1, (8, 8, 8, 16), 4, 1, 0), (1, (16, 16, 16, 16), 1, 1, 0),
    (3, (2, 2, 2, 2), 4, 8, 8), (3, (8, 8, 8, 12), 1, 8, 8), (3, (8, 8, 8, 16), 1, 8, 8),
    (3, (10, 6, 14, 12), 1, 4, 8), (3, (8, 8, 8, 16), 2, 4, 8), (3, (10, 10, 10, 20), 1, 4, 8),
    (3, (8, 8, 8, 16), 3, 2, 16), (3, (8, 8, 8, 16), 4, 2, 16)])
def test_shape_by_size(prec, dims, n, groups, pairs):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    U = synth.gauge_links(dims, 0.3, 81)
    v = synth.gaussian_source(dims, 82, nvec=n).reshape((n,) + tuple(reversed(dims)) + (4, 3))
    for variant in (-1, 0):
        c = ctx(dims, U, n_poles=20, a=0.1, b=2.7, wilson_variant=variant)
        c.sign_apply(v, np.zeros_like(v), eta=1e-5, prec=prec)
        one, stepped, g, t = c.lanczos_cycles()
        c.close()
        if variant == 0:
            assert one == 0 and stepped > 0 and g == 0
        elif sms == SMS:
            assert stepped == 0 and one > 0 and (g, t) == (groups, _tiles(dims, n, pairs, sms)[1])


def test_two_threads_with_launches_of_different_size():
    """8^4 and 8^3 x 12 run the same kernel with 2 and 3 tiles per block (49 and 74 KB of shared memory)."""
    jobs = []
    for dims in ((8, 8, 8, 8), (8, 8, 8, 12)):
        c = ctx(dims, synth.gauge_links(dims, 0.3, 81), n_poles=20, a=0.1, b=2.7)
        v = synth.gaussian_source(dims, 83)
        want = np.zeros_like(v)
        c.sign_apply(v, want, eta=1e-9, prec=3)
        jobs.append((c, v, want, []))

    def work(c, v, want, bad):
        for _ in range(40):
            o = np.zeros_like(v)
            c.sign_apply(v, o, eta=1e-9, prec=3)
            if not np.array_equal(o, want):
                bad.append(float(np.max(np.abs(o - want))))

    ts = [threading.Thread(target=work, args=j) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for c, _, _, bad in jobs:
        one, stepped, _, _ = c.lanczos_cycles()
        c.close()
        assert not bad and stepped == 0 and one == 41
