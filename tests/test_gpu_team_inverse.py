"""Inverses and log-determinants of N <= 32 by four warps a matrix: bit for bit those of one warp (whose
own test holds them to numpy), at the edges of the register widths and of the warps' shares, with
singular and non-finite matrices between good ones, and at both sides of the count that chooses."""
import numpy as np
import pytest

from test_gpu_warp_inverse import matrices, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inverse", [True, False])
@pytest.mark.parametrize("N", [1, 2, 3, 5, 8, 9, 13, 16, 17, 19, 23, 24, 25, 31, 32])
def test_equals_one_warp(N, inverse):
    S = matrices(N, 9, N)
    S[3] *= 1e-200
    S[4] = np.eye(N)[np.random.default_rng(N).permutation(N)]
    one, team = run(S, 4, inverse), run(S, 5, inverse)
    assert one[0] == 0 and team[0] == 0
    assert np.array_equal(one[1], team[1]) and np.array_equal(one[2], team[2])


@pytest.mark.parametrize("N", [6, 23, 32])
@pytest.mark.parametrize("col", [0, 1, 5, -1])
def test_singular_and_nonfinite(N, col):
    S = matrices(N, 3, 3 * N)
    for value, code in ((0.0, -5), (np.nan, -4)):
        S[1][:, col] = value
        one, team = run(S, 4), run(S, 5)
        assert one[0] == code and team[0] == code
        assert np.array_equal(one[1][[0, 2]], team[1][[0, 2]]) and np.array_equal(one[2], team[2])


@pytest.mark.parametrize("count", [1, 607, 608, 609])
def test_counts_around_the_choice(count):
    S = np.concatenate([matrices(20, 40, 7)] * 16)[:count]
    for inverse in (True, False):
        a, b = run(S, 0, inverse), run(S, 4, inverse)
        assert a[0] == 0 and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])
