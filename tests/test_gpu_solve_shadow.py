"""BiCGStab on differences of two unit sources: its shadow residual is one fixed vector,
which such a source meets in two entries only.  They take the updates of single unit
sources, or one more; those that BiCGStab gives up (four updates without progress) and
CGNE solves again report the updates of both."""
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


def test_differences_of_unit_sources(dl):
    L, T, n, tol = 8, 8, 64, 1e-10
    ctx = dl.Context(L, T, 0, 0)
    ctx.dlma_set_gauge(synth.gauge_field(L, T, 0.2, 641))
    ctx.dlma_set_params(0.05, 1.0)
    s = np.arange(L ** 3 * T)
    even = s[(s % L + s // L % L + s // L ** 2 % L + s // L ** 3) % 2 == 0]
    rng = np.random.Generator(np.random.PCG64(642))
    one = np.zeros((n, L ** 3 * T, 4, 3), dtype=np.complex128)
    two = np.zeros_like(one)
    for j in range(n):
        x, y = rng.choice(even, 2, replace=False)
        one[j, x, j % 4, j % 3] = two[j, x, j % 4, j % 3] = 1.0
        two[j, y, j % 4, j % 3] = -1.0
    ups = []
    for b in (one, two):
        _, info = ctx.dlma_solve(b, tol, dl.FP32)
        assert all(i["converged"] for i in info)
        ups.append([i["iters_outer"] for i in info])
    assert max(ups[1]) <= max(ups[0]) + 1, (max(ups[0]), sorted(ups[1])[-20:])
    ctx.close()
