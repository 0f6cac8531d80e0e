"""Tensor-core projection of values whose 8-bit digits are all near +127 with one sign, so
that the sums of the last two digit classes leave the integers that FP32 holds exactly
(2^24).  X = sum_i d_i 256^(5 - i) with d = (100, 127, 127, 127, 127, 127), x = X 2^-47 in
[1/2, 1), as real and imaginary part of every entry: c = n (1 + i)(1 - i) x^2 = 2 n x^2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
D = (100, 127, 127, 127, 127, 127)


@pytest.fixture(scope="module")
def dl():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2201_09729_gb300 as dl
    return dl


def test_aligned_digits(dl):
    L, T, N, nrhs = 8, 2, 3, 2
    n = 3 * L ** 3
    X = sum(d * 256 ** (5 - i) for i, d in enumerate(D))
    x = X * 2.0 ** -47                         # 47 bits: exact
    chunk = 256 * (2 * 100 * 127 + 3 * 127 ** 2), 256 * (2 * 100 * 127 + 4 * 127 ** 2)
    assert chunk[0] > 2 ** 24 and chunk[1] > 2 ** 24      # classes 4 and 5, 256 reals
    ctx = dl.Context(L, T, 0, 0)
    V = np.full((T, N, L ** 3, 3), x + 1j * x)
    psi = np.full((nrhs, L ** 3 * T, 4, 3), x + 1j * x)
    c = ctx.dlma_project(-1, V, psi)
    ctx.close()
    want = float(2 * n * X * X) * 2.0 ** -94
    # per product x^2: the dropped pairs of digits, i + j >= 6, at weight 2^(-14 - 8 (i + j));
    # the class sums above 2^24, 80 accumulations (class 5: 96) of at most 2 units of
    # 2^(-14 - 8 c) per chunk of 256 products; double-float sums (2^-46 of the result)
    drop = sum(D[i] * D[j] * 2.0 ** (-14 - 8 * (i + j)) for i in range(6) for j in range(6) if i + j >= 6)
    cls = (80 * 2 * 2.0 ** -46 + 96 * 2 * 2.0 ** -54) / 256
    tol = (drop + cls) / x ** 2 + 2.0 ** -46
    assert np.all(np.abs(c.real - want) <= tol * want) and np.all(np.abs(c.imag) <= tol * want)
