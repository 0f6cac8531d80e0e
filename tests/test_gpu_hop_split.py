"""FP64 operator calls on few (even site, right-hand side) pairs take the stencil that
splits a pair over 16 threads and works on the caller's arrays in place; larger batches
take the one-thread form.  Both against the oracle on either side of the switch, at site
counts that leave the last block ragged, and with overlapping input and output."""
import ctypes as C

import numpy as np
import pytest

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu
TOL = 1e-13          # FP64 rounding of about 2000 operations per site


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


# (even sites) x nrhs: 16 x 3, 252 x 1, 1080 x 11 = 11880 split, 1080 x 12 = 12960 not
@pytest.mark.parametrize("L,T,bc,nrhs", [(2, 4, 1, 3), (6, 2, 0, 1), (6, 10, 1, 11), (6, 10, 1, 12)])
def test_operator_both_forms(dl, L, T, bc, nrhs):
    m0, csw = 0.15, 1.1
    U = synth.gauge_field(L, T, 0.25, 611)
    ctx = dl.Context(L, T, bc, 0)
    ctx.dlma_set_gauge(U)
    ctx.dlma_set_params(m0, csw)
    eo = dirac.EvenOdd(U, L, T, m0, csw, bc)
    V = L ** 3 * T
    psi = synth.gaussian_spinors(nrhs, V, 612)
    he = np.ascontiguousarray(psi[:, :V // 2])

    def close(got, want):
        assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)

    close(ctx.dlma_apply_Dw(psi, dl.FP64), eo.apply_full(psi))
    close(ctx.dlma_apply_schur(he, 0, dl.FP64), eo.schur(he))
    close(ctx.dlma_apply_schur(he, 1, dl.FP64), eo.schur_dag(he))
    torch = pytest.importorskip("torch")
    buf = torch.from_numpy(he.copy()).cuda()
    p = C.c_void_p(buf.data_ptr())
    assert ctx.lib.dlma_apply_schur(ctx.h, p, p, nrhs, 0, dl.FP64, 1) == 0       # in place
    close(buf.cpu().numpy(), eo.schur(he))
    x, info = ctx.dlma_solve(psi[:2], 1e-12, dl.FP64)                            # fused CG epilogue, norms
    assert all(i["converged"] for i in info)
    close_r = np.linalg.norm(eo.apply_full(x) - psi[:2]) / np.linalg.norm(psi[:2])
    assert close_r <= 1e-12
    ctx.close()
