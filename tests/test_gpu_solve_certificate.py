"""The residual that a mixed-precision solve reports, and on which it calls a right-hand
side converged, against b - D x of the oracle: systems close to the critical mass (on this
4^4 field the even-odd operator's condition number is 1.7e1 at m0 = 0.08, 2.8e3 at -0.08
and 1.9e4 at -0.082) and tolerances down to the rounding level of FP64."""
import numpy as np
import pytest

import synth
from oracle import dirac

pytestmark = pytest.mark.gpu
L, T, CSW, NRHS = 4, 4, 1.0, 5


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


def check(ctx, dl, eo, b, prec, tols):
    for tol in tols:
        x, info = ctx.dlma_solve(b, tol, getattr(dl, prec), allow_not_converged=True)
        for j in range(NRHS):
            nb = np.linalg.norm(b[j].ravel())
            r = np.linalg.norm((b[j] - eo.apply_full(x[j])).ravel()) / nb
            # rounding of b - D x itself: 2^-53 of |T| + 8 |hop| = 4.7 + 8 sqrt 3 < 19 times
            # |x| for each of the two evaluations, the oracle's and the library's
            noise = 2 * 2.0 ** -53 * 19 * np.linalg.norm(x[j].ravel()) / nb
            got = info[j]["true_resid"]
            assert abs(got - r) <= 0.05 * r + 0.025 * tol + noise, (tol, j, got, r, noise)
            if info[j]["converged"]:
                assert r <= 1.05 * tol + noise, (tol, j, got, r)


@pytest.mark.parametrize("m0", [0.08, -0.08, -0.082])
@pytest.mark.parametrize("prec,solver", [("FP32", "SOLVER_BICGSTAB"), ("FP32", "SOLVER_CGNE"), ("FP16S", "SOLVER_CGNE")])
def test_reported_residual(dl, m0, prec, solver):
    U = synth.gauge_field(L, T, 0.2, 701)
    eo = dirac.EvenOdd(U, L, T, m0, CSW)
    b = synth.gaussian_spinors(NRHS, L ** 3 * T, 702)
    ctx = dl.Context(L, T, 0, 0)
    ctx.dlma_set_gauge(U)
    ctx.dlma_set_params(m0, CSW)
    ctx.dlma_set_solver(getattr(dl, solver))
    check(ctx, dl, eo, b, prec, (1e-8, 1e-10, 1e-12, 1e-13, 1e-14, 2e-15, 3e-16))
    ctx.close()


@pytest.mark.parametrize("prec,solver", [("FP32", "SOLVER_BICGSTAB"), ("FP32", "SOLVER_CGNE"), ("FP16S", "SOLVER_CGNE")])
def test_links_off_su3(dl, prec, solver, monkeypatch):
    # third rows 1e-4 off: the 12-real FP32 links rebuild other ones than FP64 reads
    monkeypatch.setenv("DLMA_FORCE_LINKS", "12")
    rng = np.random.Generator(np.random.PCG64(703))
    U = synth.gauge_field(L, T, 0.2, 701)
    U[..., 2, :] += 1e-4 * (rng.standard_normal(U[..., 2, :].shape) + 1j * rng.standard_normal(U[..., 2, :].shape))
    eo = dirac.EvenOdd(U, L, T, 0.08, CSW)
    b = synth.gaussian_spinors(NRHS, L ** 3 * T, 702)
    ctx = dl.Context(L, T, 0, 0)
    ctx.dlma_set_gauge(U)
    ctx.dlma_set_params(0.08, CSW)
    ctx.dlma_set_solver(getattr(dl, solver))
    check(ctx, dl, eo, b, prec, (1e-8, 1e-10))
    ctx.close()
