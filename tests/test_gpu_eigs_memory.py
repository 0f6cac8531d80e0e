"""The eigensolve with little device memory left: the digit buffers of the tensor-core
products (2.5 GB for this block) do not fit, the other buffers do."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


def test_eigs_without_room_for_digits(dl):
    torch = pytest.importorskip("torch")
    L, T, N = 16, 32, 32
    ctx = dl.Context(L, T, 0, 0)
    ctx.dlma_set_gauge(synth.gauge_field(L, T, 0.2, 651))
    want, _ = ctx.dlma_laplacian_eigs(-1, N, 1e-10, want_vecs=False)
    ctx.dlma_release_workspace()
    torch.cuda.empty_cache()
    # blocks 4 x 0.2 + 3 x 0.4 GB, cached modes 0.2 GB, small ones: 2.4 GB
    left = 3_400_000_000
    free, _ = torch.cuda.mem_get_info()
    hog = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    try:
        got, _ = ctx.dlma_laplacian_eigs(-1, N, 1e-10, want_vecs=False)
    finally:
        del hog
        torch.cuda.empty_cache()
        ctx.close()
    # both to residuals of 1e-10: eigenvalues of a hermitian operator to that, twice
    assert np.abs(got - want).max() <= 2e-10 * 12
