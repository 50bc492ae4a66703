"""A product of which only parts fit the workspace of the tensor-core form, added to what C and D hold: each
part is added once, whether it runs in that form or by the tiles."""
import numpy as np
import pytest

from test_gpu_gemm_slices import N_, gemm, long_product, rand

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ws", [0, 1 << 10, 9 << 10, 20 << 10, 60 << 10, 100 << 10, 200 << 10])
@pytest.mark.parametrize("m,n,k", [(1, 1, 5120), (1, 1, 20000), (2, 3, 8000), (1, 5, 700)])
def test_parts_are_added_once(m, n, k, ws):
    rng = np.random.default_rng(k + m)
    for ar, br in ((0, 0), (1, 0), (1, 1)):
        A, B, C, D = rand(rng, ar, m, k), rand(rng, br, k, n), rand(rng, 0, m, n), rand(rng, 0, m, n)
        for form in (1, 2):
            got, Dg, _, _ = gemm(A, B, C, m, n, k, a=(ar, N_, k, (0, 0, 0)), b=(br, N_, n, (0, 0, 0)), ldc=n, beta=1.0, D=D,
                                 ldd=n, form=form, ws=ws)
            re, im = long_product(A, B)
            want = np.asarray(re, float) + 1j * np.asarray(im, float) + C
            tol = 2.0 ** -50 * np.sqrt(k) * 4 + 1e-14 * np.sqrt(k)
            assert np.max(np.abs(got - want)) < tol and np.max(np.abs(Dg - D - want)) < tol
