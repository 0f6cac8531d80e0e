"""Orthonormality of the Laplacian modes: the arithmetic that the eigensolver picks for its
FP64-accurate products (double-float or the tensor cores' digits) leaves them no worse than
double-float does."""
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


# sums over few rows (small timeslices, few of them, few columns), and the two last sizes,
# where the tensor cores take over
@pytest.mark.parametrize("L,T,N", [(8, 20, 24), (10, 18, 20), (10, 18, 32), (12, 12, 22), (14, 12, 32), (16, 32, 16),
                                   (16, 16, 32), (12, 24, 48)])
def test_modes_no_worse_than_double_float(dl, L, T, N, monkeypatch):
    torch = pytest.importorskip("torch")
    U = synth.gauge_field(L, T, 0.2, 671)
    rms = {}
    for tc in ("0", None):
        if tc is None:
            monkeypatch.delenv("DLMA_EIGS_TC", raising=False)
        else:
            monkeypatch.setenv("DLMA_EIGS_TC", tc)
        ctx = dl.Context(L, T, 0, 0)
        ctx.dlma_set_gauge(torch.from_numpy(U).cuda())
        _, V = ctx.dlma_laplacian_eigs(-1, N, 1e-10, device_out=True)
        V = V.reshape(T, N, -1)
        d = V.conj() @ V.transpose(1, 2) - torch.eye(N, dtype=V.dtype, device=V.device)
        rms[tc] = float(d.abs().square().mean().sqrt())
        ctx.close()
    # 10 % for the different path of the two iterations
    assert rms[None] <= 1.1 * rms["0"], rms
