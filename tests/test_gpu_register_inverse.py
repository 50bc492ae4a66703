"""The register Gauss-Jordan kernel (32 < N <= 128) at the edges of its panels of four columns, of its
groups of warps and of its two CTAs, in FP64 and in float pairs: inverses and log-determinants against
numpy, permutations (exact), entries outside the range of the integer conversions, and a zero or
non-finite column at each place of a panel."""
import numpy as np
import pytest

from oracle import afqmc as O
from paper_2003_01831_gb300 import api
from test_gpu_warp_inverse import matrices, run

pytestmark = pytest.mark.gpu
EPS = {2: 1e-15, 3: 2.0**-44}   # variant 2: FP64, 3: float pairs


@pytest.mark.parametrize("variant", [2, 3])
@pytest.mark.parametrize("N", [33, 34, 36, 37, 47, 61, 63, 64, 65, 66, 68, 95, 97, 126, 127, 128])
def test_inverse_and_logdet(N, variant):
    S = matrices(N, 5, N)
    kappa = max(np.linalg.cond(s) for s in S)
    ref = O.log_det(S)
    rc, X, ld, _ = run(S, variant)
    assert rc == 0, api.afqmc_last_error()
    # elimination with pivoting: a few N kappa roundings
    tol = EPS[variant] * 10 * N * kappa
    assert np.max(np.abs(S @ X - np.eye(N))) < tol
    assert np.max(np.abs(X - np.linalg.inv(S))) < tol * np.max(np.abs(X))
    assert np.max(np.abs(ld.real - ref.real)) < tol
    assert np.max(np.abs(np.angle(np.exp(1j * (ld.imag - ref.imag))))) < tol


@pytest.mark.parametrize("variant", [2, 3])
@pytest.mark.parametrize("N", [40, 64, 101, 128])
def test_scaled_permutations_are_exact(N, variant):
    """Powers of two in permuted places, some so small that a float pair's conversion leaves the
    normal range of its low half: every product and reciprocal is exact."""
    rng = np.random.default_rng(N)
    e = rng.integers(-100, 100, size=(4, N))
    P = np.zeros((4, N, N), dtype=np.complex128)
    for b in range(4):
        P[b, np.arange(N), rng.permutation(N)] = np.ldexp(1.0, e[b]) * np.array([1, -1, 1j, -1j])[rng.integers(0, 4, N)]
    rc, X, ld, _ = run(P, variant)
    assert rc == 0
    ref = np.zeros_like(P)
    nz = P != 0
    ref[nz] = 1.0 / P[nz]
    assert np.array_equal(X, np.swapaxes(ref, 1, 2))
    for b in range(4):
        assert abs(ld[b].real - np.sum(e[b]) * np.log(2.0)) < 1e-15 * 100 * N * np.log(2.0)


@pytest.mark.parametrize("variant", [2, 3])
@pytest.mark.parametrize("N", [35, 64, 98, 128])
@pytest.mark.parametrize("col", [0, 1, 2, 3, 4, 33, -1])
def test_singular_and_nonfinite_columns(N, variant, col):
    S = matrices(N, 3, 7 * N)
    good = run(S[:1], variant)[1]
    S[1][:, col] = 0.0
    rc, X, ld, _ = run(S, variant)
    assert rc == -5
    assert np.array_equal(X[0], good[0]) and np.isneginf(ld[1].real) and np.all(np.isfinite(ld[[0, 2]]))
    S[1][:, col] = np.nan
    rc, X, ld, _ = run(S, variant)
    assert rc == -4
    assert np.array_equal(X[0], good[0]) and np.isneginf(ld[1].real) and np.all(np.isfinite(ld[[0, 2]]))
