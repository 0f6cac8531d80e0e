"""FP32 on pairs of right-hand sides (large batches): odd batches just above the switches,
the operator against FP64, BiCGStab with a zero source and a repeated one against the
single-vector form."""
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


def test_pairs_and_single(dl):
    torch = pytest.importorskip("torch")
    L, T, nrhs, tol = 8, 16, 257, 1e-10           # 257 x 4096 even sites: above 2^20
    ctx = dl.Context(L, T, 1, 0)
    ctx.dlma_set_gauge(synth.gauge_field(L, T, 0.2, 631))
    ctx.dlma_set_params(0.08, 1.1)
    V, Vs = L ** 3 * T, L ** 3
    b = torch.zeros((nrhs, V, 4, 3), dtype=torch.complex128, device="cuda")
    b[:, :Vs] = torch.from_numpy(synth.z2z2_noise(nrhs, Vs, 632)).cuda()
    b[5] = 0
    b[nrhs - 1] = b[0]                             # the last vector has an empty partner
    x, info = ctx.dlma_solve(b, tol, dl.FP32)
    assert all(i["converged"] for i in info)
    r = torch.linalg.vector_norm((b - ctx.dlma_apply_Dw(x, dl.FP64)).flatten(1), dim=1)
    n = torch.linalg.vector_norm(b.flatten(1), dim=1)
    assert bool((r <= tol * n).all()) and not bool(x[5].any())
    # solved to a residual of 1e-10 either way: equal to 1e-10 times the condition (< 1e2)
    one, _ = ctx.dlma_solve(b[:1].contiguous(), tol, dl.FP32)
    for y in (x[0], x[nrhs - 1]):
        assert float(torch.linalg.vector_norm(y - one[0]) / torch.linalg.vector_norm(one[0])) < 1e-8
    ctx.close()


def test_operator_pairs(dl):
    torch = pytest.importorskip("torch")
    L, T, nrhs = 8, 16, 27                         # 27 x 4096 even sites: above 10^5
    ctx = dl.Context(L, T, 1, 0)
    ctx.dlma_set_gauge(synth.gauge_field(L, T, 0.25, 633))
    ctx.dlma_set_params(0.1, 1.2)
    V = L ** 3 * T
    psi = torch.from_numpy(synth.gaussian_spinors(nrhs, V, 634)).cuda()
    he = psi[:, :V // 2].contiguous()
    for got, want in [(ctx.dlma_apply_Dw(psi, dl.FP32), ctx.dlma_apply_Dw(psi, dl.FP64)),
                      (ctx.dlma_apply_schur(he, 0, dl.FP32), ctx.dlma_apply_schur(he, 0, dl.FP64)),
                      (ctx.dlma_apply_schur(he, 1, dl.FP32), ctx.dlma_apply_schur(he, 1, dl.FP64))]:
        d = torch.linalg.vector_norm((got - want).flatten(1), dim=1)
        assert bool((d < 1e-6 * torch.linalg.vector_norm(want.flatten(1), dim=1)).all())
    ctx.close()
