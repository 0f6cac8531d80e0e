"""Tensor-core projection where its work is cut differently: one or several blocks per
tile (chunks of kappa shared out), one or several chunk groups (bounded digit buffers),
ragged rows, modes and last chunk.  Against numpy, relative to the row and mode norms."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
TOL = 1e-12          # digits to 2^-48 of a chunk's largest entry, products to 2^-47


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


# chunks of 128 kappa: 2 (one block per tile), 14 (last one of 20 kappa; few tiles),
# 41 (many blocks per tile); the cap of 64 MB cuts the last into several groups
@pytest.mark.parametrize("L,T,N,nrhs,cap", [(4, 4, 1, 1, 0), (8, 2, 33, 33, 0), (12, 2, 5, 3, 0),
                                            (12, 4, 33, 40, 64 << 20)])
def test_projection(dl, L, T, N, nrhs, cap):
    ctx = dl.Context(L, T, 0, 0)
    if cap:
        ctx.dlma_set_memory_cap(cap)
    rng = np.random.Generator(np.random.PCG64(811))
    n = 3 * L ** 3
    V = rng.standard_normal((T, N, n)) + 1j * rng.standard_normal((T, N, n))
    psi = synth.gaussian_spinors(nrhs, L ** 3 * T, 812)
    psi *= 10.0 ** rng.uniform(-3, 3, (nrhs, L ** 3 * T, 1, 1))
    torch = pytest.importorskip("torch")       # device arrays: the cap bounds the library's buffers only
    c = ctx.dlma_project(-1, torch.from_numpy(V.reshape(T, N, L ** 3, 3)).cuda(), torch.from_numpy(psi).cuda())
    c = c.cpu().numpy()
    p = psi.reshape(nrhs, T, L ** 3, 4, 3).transpose(0, 1, 3, 2, 4).reshape(nrhs, T, 4, n)
    want = np.einsum("jtan,tkn->jtak", p, V.conj(), optimize=True)
    scale = np.linalg.norm(p, axis=-1)[..., None] * np.linalg.norm(V, axis=-1)[None, :, None, :]
    assert np.all(np.abs(c - want) <= TOL * scale)
    ctx.close()
