"""FP64 products with an output's contraction shared by four or eight threads: every operand form, K
below, at and past the threads' shares, batches, beta and a second output, against long double sums."""
import itertools

import numpy as np
import pytest

from test_gpu_gemm_slices import C_, N_, T_, gemm, long_product, op_of, rand

pytestmark = pytest.mark.gpu


def check(got, A, B, k):
    """One rounding a product and a sum: (k + 8) 2^-52 of the sum of the products' sizes."""
    re, im = long_product(A, B)
    size = np.abs(A) @ np.abs(B)
    assert np.all(np.hypot(np.asarray(got.real - re, dtype=float), np.asarray(got.imag - im, dtype=float))
                  <= (k + 8) * 2.0 ** -52 * size)


@pytest.mark.parametrize("form", [4, 5])
@pytest.mark.parametrize("ar,br", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (3, 5, 7), (1, 9, 8), (5, 2, 15), (24, 5, 24), (7, 11, 31), (2, 3, 32),
                                   (9, 4, 33), (5, 5, 120), (3, 2, 513)])
def test_shared_contractions(form, ar, br, m, n, k):
    rng = np.random.default_rng(m * 100 + n * 10 + k)
    for opa, opb in itertools.product((N_, T_, C_), repeat=2):
        if (opa == C_ and ar) or (opb == C_ and br):
            continue
        A = rand(rng, ar, m, k) if opa == N_ else rand(rng, ar, k, m)
        B = rand(rng, br, k, n) if opb == N_ else rand(rng, br, n, k)
        kw = dict(a=(ar, opa, A.shape[1], (0, 0, 0)), b=(br, opb, B.shape[1], (0, 0, 0)), ldc=n)
        C, D = rand(rng, 0, m, n), rand(rng, 0, m, n)
        got, second, _, _ = gemm(A, B, C, m, n, k, form=form, D=D, ldd=n, **kw)
        check(got, op_of(A, opa), op_of(B, opb), k)
        assert np.array_equal(second, D + got)
        again = gemm(A, B, C, m, n, k, form=form, alpha=2.0, beta=1.0, **kw)[0]
        assert np.max(np.abs(again - (2.0 * got + C))) <= 2.0 ** -50 * np.max(np.abs(2.0 * got) + np.abs(C))


@pytest.mark.parametrize("W", [1, 3, 16, 61])
def test_batches_and_choice(W):
    rng = np.random.default_rng(W)
    M, N = 24, 5
    Psi, Phi = rand(rng, 0, M, N), rand(rng, 0, W, M, N)
    S = np.full((W, N, N), np.nan + 0j)
    for form in (2, 4, 5):
        got, _, chose, _ = gemm(Psi, Phi, S, N, N, M, nb=(W, 1, 1), a=(0, C_, N, (0, 0, 0)), b=(0, N_, N, (M * N, 0, 0)),
                                ldc=N, sc=(N * N, 0, 0), form=form, ws=0)
        check(got, np.conj(Psi.T)[None], Phi, M)
        assert chose == 4
