"""The one-warp Gauss-Jordan kernel (N <= 32) against numpy: every register width (8, 16, 24, 32
columns) at its edges, a matrix count that leaves the last CTA half empty, log-determinants alone,
permutations (exact), and singular and non-finite matrices beside good ones."""
import ctypes

import numpy as np
import pytest

from oracle import afqmc as O
from paper_2003_01831_gb300 import api

pytestmark = pytest.mark.gpu


def run(S, variant=0, with_inverse=True):
    L = api.lib()
    vp = ctypes.c_void_p
    L.afqmc_debug_inverse.restype = ctypes.c_int
    L.afqmc_debug_inverse.argtypes = [vp, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int, vp, vp, vp]
    S = np.ascontiguousarray(S, dtype=np.complex128)
    count, N, _ = S.shape
    X, ld, ms = np.zeros_like(S), np.zeros(count, dtype=np.complex128), ctypes.c_float(0.0)
    rc = L.afqmc_debug_inverse(S.ctypes.data, N, count, variant, int(with_inverse), X.ctypes.data, ld.ctypes.data,
                               ctypes.addressof(ms))
    return rc, X, ld, ms.value


def matrices(N, count, seed):
    rng = np.random.default_rng(seed)
    return np.eye(N) + 0.7 * (rng.standard_normal((count, N, N)) + 1j * rng.standard_normal((count, N, N))) / np.sqrt(N)


@pytest.mark.parametrize("N", [1, 2, 7, 8, 9, 15, 16, 17, 24, 25, 31, 32])
def test_inverse_and_logdet(N):
    S = matrices(N, 5, N)
    kappa = max(np.linalg.cond(s) for s in S)
    ref = O.log_det(S)
    rc, X, ld, _ = run(S)
    assert rc == 0, api.afqmc_last_error()
    # elimination with pivoting in FP64: a few N kappa roundings
    assert np.max(np.abs(S @ X - np.eye(N))) < 1e-15 * 10 * N * kappa
    assert np.max(np.abs(X - np.linalg.inv(S))) < 1e-15 * 10 * N * kappa * np.max(np.abs(X))
    rc, _, l2, _ = run(S, with_inverse=False)
    assert rc == 0
    for got in (ld, l2):
        assert np.max(np.abs(got.real - ref.real)) < 1e-13 * N
        assert np.max(np.abs(np.angle(np.exp(1j * (got.imag - ref.imag))))) < 1e-13 * N


@pytest.mark.parametrize("N", [3, 8, 20, 32])
def test_permutations_are_exact(N):
    rng = np.random.default_rng(N)
    P = np.stack([np.eye(N)[rng.permutation(N)] for _ in range(6)] + [np.eye(N)[::-1]]).astype(np.complex128)
    rc, X, ld, _ = run(P)
    assert rc == 0
    assert np.array_equal(X, np.swapaxes(P, 1, 2))
    sign = np.linalg.det(P.real)
    assert np.array_equal(ld.real, np.zeros(len(P)))
    assert np.max(np.abs(np.exp(1j * ld.imag) - sign)) < 1e-15 * 4


@pytest.mark.parametrize("N", [6, 32])
def test_singular_and_nonfinite(N):
    for kind, code in (("zero column", -5), ("nan", -4), ("inf", -4)):
        S = matrices(N, 3, 3)
        if kind == "zero column":
            S[1][:, N - 2] = 0.0
        elif kind == "nan":
            S[1][2, 1] = np.nan
        else:
            S[1][:, 0] = np.inf
        for inv in (True, False):
            rc, X, ld, _ = run(S, with_inverse=inv)
            assert rc == code, (kind, rc)
            assert ld[1].real == -np.inf
            ref = O.log_det(S[[0, 2]])
            assert np.max(np.abs(ld[[0, 2]].real - ref.real)) < 1e-13 * N
        if kind == "zero column":
            rc, X, ld, _ = run(S)
            assert np.max(np.abs(S[2] @ X[2] - np.eye(N))) < 1e-12 * N
