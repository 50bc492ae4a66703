"""The Cholesky QR of mixed walker sets on walkers of very large and very small norms (M < 2 N: the Gram
matrices are formed in FP64): orthonormal columns as for walkers of norm one."""
import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


# tolerances: float pairs (2^-44, times N and a squared condition of about 10); at 2^-65 the Gram matrix's
# entries near 2^-130 are held to 2^-149, 2^-19 of them, times N
@pytest.mark.parametrize("p,tol", [(0, 1e-9), (40, 1e-9), (62, 1e-9), (-40, 1e-9), (-65, 40 * 2.0 ** -17)])
def test_norms_across_the_float_range(p, tol):
    rng = np.random.default_rng(3)
    M, N, W = 64, 40, 3
    h, L, E0 = syn.make_hamiltonian(M, 64, rng)
    Psi = syn.make_trial(h, N, N)
    F = Psi[0][None] + 0.05 * (rng.standard_normal((W, M, N)) + 1j * rng.standard_normal((W, M, N)))
    F = F * 2.0 ** p
    with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, Phi0=(F, F), k_qr=1, precision=api.PREC_BF16X3) as g:
        g.step(1, seed=4)
        for Q in g.walkers()[:2]:
            for w in range(W):
                assert np.max(np.abs(Q[w].conj().T @ Q[w] - np.eye(N))) < tol
