"""The Cholesky factor's inverse of the tensor-core QR at the edges of its kernels' sizes (32, 64, 128
columns and the multiples of 8 around them): after a step that re-orthonormalises, every walker's columns
are orthonormal and span what they did without it; a dead walker keeps its orbitals."""
import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 24, 32, 40, 64, 72, 96, 128])
def test_orthonormal_columns_of_the_same_span(N):
    rng = np.random.default_rng(N)
    M, nch, W = max(64, (2 * N + 63) // 64 * 64), 64, 5
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    amp = 0.8 / np.sqrt(M)
    Phi0 = [Psi[s][None] + amp * (rng.standard_normal((W, M, N)) + 1j * rng.standard_normal((W, M, N))) for s in range(2)]
    out = {}
    for k_qr in (0, 1):
        with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, Phi0=Phi0, k_qr=k_qr, precision=api.PREC_BF16X3) as g:
            Pu, Pd, w, step = g.walkers()
            w[2] = 0.0
            g.set_walkers(Pu, Pd, w, step)
            g.step(1, seed=4)
            out[k_qr] = g.walkers()[:2]
    for s in range(2):
        for w in range(W):
            P, Q = out[0][s][w], out[1][s][w]
            if w == 2:   # through the three-slice product with the identity
                assert np.max(np.abs(P - Q)) < 10 * N * 2.0 ** -30 * np.max(np.abs(P))
                continue
            # three fp16 slices an operand (2^-30 of its rows' norms), squared condition ~10
            assert np.max(np.abs(Q.conj().T @ Q - np.eye(N))) < 10 * N * 2.0 ** -30
            R = Q.conj().T @ P
            assert np.max(np.abs(P - Q @ R)) < 10 * N * 2.0 ** -30 * np.max(np.abs(P))
            assert np.max(np.abs(np.tril(R, -1))) < 10 * N * 2.0 ** -30 * np.max(np.abs(R))
