"""The waits of the tensor-core Gram kernel when their time runs out. Lanes poll for themselves, so
a warp must agree on the outcome before anything that takes it as one; read from the source: the
plain wait is used by the voting wait and by the one thread that drains the MMAs, nowhere else.
On the GPU a limit of zero gives up everywhere and a very short one anywhere: the call ends with
OVL_ETIMEOUT (or, when nothing gave up, the right block) and the context stays usable."""
import os
import re

import numpy as np
import pytest

import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_01855_gb300", "csrc")


def test_warps_vote_on_every_wait():
    with open(os.path.join(CSRC, "tcgram.cu")) as f:
        src = re.sub(r"//.*", "", f.read())
    calls = [m.group(0) for m in re.finditer(r"\bmbar_wait\(smem_u32[^;]*;|\bmbar_wait\(bar[^;]*;", src)]
    assert sorted(calls) == ["mbar_wait(bar, parity, gave_up, limit);",
                             "mbar_wait(smem_u32(&drain), 0u, nullptr, TG_DRAIN_NS);"]
    body = src[src.index("bool warp_wait("):]
    assert "__all_sync(0xffffffffu, ok)" in body[:body.index("}")]
    assert len(re.findall(r"\bwarp_wait\(smem_u32", src)) == 4


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
def test_gram_wait_that_runs_out(prec):
    from tests.gpu_util import ctx, lib
    B = lib()
    dims = (8, 8, 4, 4)
    c = ctx(dims, synth.unit_links(dims), a=0.2, b=2.6)
    rng = np.random.default_rng(3)
    shp = (70,) + tuple(reversed(dims)) + (4, 3)
    A = (rng.standard_normal(shp) + 1j * rng.standard_normal(shp)).astype(np.complex128 if prec == 0 else np.complex64)
    A2 = A.reshape(70, -1).astype(np.complex128)
    ref = np.conj(A2) @ A2.T
    scale = np.outer(np.linalg.norm(A2, axis=1), np.linalg.norm(A2, axis=1))
    for limit in (0.0, 1e-7, 1e-6, 3e-6, 1e-5):
        c.set_wait_limit(limit)
        try:
            G = c.gram(A, A, prec=prec)
        except B.OvlError as e:
            assert e.status == B.OVL_ETIMEOUT
        else:
            assert limit > 0 and np.max(np.abs(G - ref) / scale) <= 1e-12
    c.set_wait_limit(2.0)
    assert np.max(np.abs(c.gram(A, A, prec=prec) - ref) / scale) <= 1e-12
    for bad in (-1.0, 3601.0, float("nan")):
        with pytest.raises(B.OvlError):
            c.set_wait_limit(bad)
