"""Long vectors in a Gram block of so many tiles that every block of the launch sums whole vectors by
itself (640 x 640: 100 tiles, one split; 3072 exact chunks each): diagonal and some off-diagonal
entries against FP64. Each chunk adds one double-float rounding, at most 2^-47 of the running sum, to an
entry; as independent errors sqrt(3072 / 3) of them are 2e-13 on the diagonal, held to 1e-12."""
import numpy as np
import pytest

import synth
from tests.gpu_util import ctx

pytestmark = pytest.mark.gpu


def test_gram_many_tiles_long_vectors():
    import torch
    dims, n = (16, 16, 16, 16), 640
    c = ctx(dims, synth.unit_links(dims), a=0.2, b=2.6)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A = torch.randn((n,) + tuple(reversed(dims)) + (4, 3), generator=g, device="cuda", dtype=torch.complex64)
    G = c.gram(A, A, prec=1)
    c.close()
    F = A.flatten(1)
    norm2 = np.array([float(torch.linalg.vector_norm(F[i].to(torch.complex128)) ** 2) for i in range(n)])
    err = np.abs(np.diag(G) - norm2) / norm2
    print("diagonal: largest relative error %.2e" % err.max())
    assert err.max() <= 1e-12
    row = (F[:1].to(torch.complex128).conj() @ F[:64].to(torch.complex128).transpose(0, 1)).cpu().numpy()[0]
    assert np.max(np.abs(G[0, :64] - row)) <= 1e-12 * norm2.max()
