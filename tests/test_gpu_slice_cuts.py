"""A contraction much longer than the workspace holds (hundreds of pieces, a few at a time) on the sliced
tensor-core form: the cuts' sums equal the product."""
import numpy as np
import pytest

from test_gpu_gemm_slices import N_, check, gemm, rand

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,ws", [(20000, 600 << 10), (100003, 900 << 10), (150000, 4 << 20)])
def test_many_cuts(k, ws):
    rng = np.random.default_rng(k)
    m, n = 24, 5
    A, B = rand(rng, 1, m, k), rand(rng, 0, k, n)
    C = np.full((m, n), np.nan + 0j)
    got = gemm(A, B, C, m, n, k, a=(1, N_, k, (0, 0, 0)), b=(0, N_, n, (0, 0, 0)), ldc=n, ws=ws)[0]
    check(got, A, B)
