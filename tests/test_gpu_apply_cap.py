"""FP32 operator calls on an odd number of right-hand sides under a memory cap that holds
exactly their vectors: the pair form, which would round the number up, is not taken."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


def test_odd_batch_at_the_cap(dl):
    torch = pytest.importorskip("torch")
    L, T, n = 8, 16, 25                        # 25 x 4096 even sites: pairs without a cap
    Vh = L ** 3 * T // 2
    ctx = dl.Context(L, T, 1, 0)
    ctx.dlma_set_gauge(synth.gauge_field(L, T, 0.2, 661))
    ctx.dlma_set_params(0.1, 1.0)
    psi = torch.from_numpy(synth.gaussian_spinors(n, 2 * Vh, 662)).cuda()
    half = psi[:, :Vh].contiguous()
    want = ctx.dlma_apply_Dw(psi, dl.FP64), ctx.dlma_apply_schur(half, 0, dl.FP64)
    for k, cap in ((0, 2 * n * 96 * Vh + 256), (1, n * 96 * Vh + 256)):
        ctx.dlma_release_workspace()
        ctx.dlma_set_memory_cap(cap)
        got = ctx.dlma_apply_schur(half, 0, dl.FP32) if k else ctx.dlma_apply_Dw(psi, dl.FP32)
        ctx.dlma_set_memory_cap(0)
        d = torch.linalg.vector_norm((got - want[k]).flatten(1), dim=1)
        assert bool((d < 1e-6 * torch.linalg.vector_norm(want[k].flatten(1), dim=1)).all())
    ctx.close()
