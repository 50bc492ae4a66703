"""FP64 products on CTA pairs (two neighbouring row tiles of the sliced tensor-core form): even and odd
numbers of row tiles, ragged last tiles and columns, one and several pieces of the contraction, batches."""
import numpy as np
import pytest

from test_gpu_gemm_slices import N_, check, gemm, rand

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ar,br", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("rows,cols,k", [(129, 33, 40), (256, 64, 128), (257, 65, 70), (1030, 20, 33), (1153, 31, 600),
                                         (1281, 64, 129)])
def test_row_tile_pairs(ar, br, rows, cols, k):
    rng = np.random.default_rng(rows + cols + k)
    for m, n in ((rows, cols), (cols, rows)):
        A, B = rand(rng, ar, m, k), rand(rng, br, k, n)
        C = np.full((m, n), np.nan + 0j)
        got = gemm(A, B, C, m, n, k, a=(ar, N_, k, (0, 0, 0)), b=(br, N_, n, (0, 0, 0)), ldc=n)[0]
        check(got, A, B)


@pytest.mark.parametrize("W,m,n,k", [(3, 200, 40, 64), (5, 300, 100, 150), (2, 1200, 30, 700)])
def test_shared_batches(W, m, n, k):
    rng = np.random.default_rng(W)
    A, B = rand(rng, 0, W, m, k), rand(rng, 0, W, k, n)
    C = np.full((W, m, n), np.nan + 0j)
    got = gemm(A, B, C, m, n, k, nb=(W, 1, 1), a=(0, N_, k, (m * k, 0, 0)), b=(0, N_, n, (k * n, 0, 0)), ldc=n,
               sc=(m * n, 0, 0))[0]
    check(got, A, B)
