"""BiCGStab on pairs of right-hand sides at batches of at most 16, which run as they come
(larger ones go through the batch-size tuner, whose choice may fall below the switch of
2^20 even sites x right-hand sides): 15 x 73728 even sites, with an empty partner, zero
sources and partners that converge at different times."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


def test_odd_batch_of_pairs(dl):
    torch = pytest.importorskip("torch")
    L, T, n, tol = 16, 36, 15, 1e-10
    V, Vs = L ** 3 * T, L ** 3
    assert n <= 16 and n * (V // 2) >= 1 << 20 and 7 * (V // 2) < 1 << 20
    ctx = dl.Context(L, T, 1, 0)
    ctx.dlma_set_gauge(torch.from_numpy(synth.gauge_field(L, T, 0.2, 681)).cuda())
    ctx.dlma_set_params(0.06, 1.1)
    b = torch.zeros((n, V, 4, 3), dtype=torch.complex128, device="cuda")
    noise = torch.from_numpy(synth.z2z2_noise(n, Vs, 682)).cuda()
    b[:, :Vs] = noise
    for j in (3, 9, 14):                       # unit sources converge after other iterations
        b[j] = 0
        b[j, 5 * j, j % 4, j % 3] = 1.0
    b[4] = 0                                   # (4, 5): an idle partner from the start
    b[6] = b[7] = 0                            # (6, 7): an idle pair
    x, info = ctx.dlma_solve(b, tol, dl.FP32)
    assert all(i["converged"] for i in info)
    r = torch.linalg.vector_norm((b - ctx.dlma_apply_Dw(x, dl.FP64)).flatten(1), dim=1)
    nb = torch.linalg.vector_norm(b.flatten(1), dim=1)
    assert bool((r <= tol * nb).all())
    for j in (4, 6, 7):
        assert not bool(x[j].any()) and info[j]["iters_inner"] == 0
    # batches of 7 (below the switch) iterate on single vectors: the same solutions to the
    # residual of 1e-10 times the condition (< 1e2), from the same recursion (the iteration
    # counts of FP32 recursions with other rounding differ by a few)
    for j0 in (0, 8):
        y, one = ctx.dlma_solve(b[j0:j0 + 7].contiguous(), tol, dl.FP32)
        for k in range(7):
            j = j0 + k
            if j in (4, 6):
                continue
            assert float(torch.linalg.vector_norm(x[j] - y[k]) / torch.linalg.vector_norm(y[k])) < 1e-8
            assert abs(info[j]["iters_inner"] - one[k]["iters_inner"]) <= 0.1 * one[k]["iters_inner"] + 2
    ctx.close()
