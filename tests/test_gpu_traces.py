"""The traces t_n = Tr T_n and X_n = Tr(T_n T_n) of the FP64 step through the local energy and the force
bias, at the electron counts where their kernel changes form (a warp, a CTA, more than shared memory
holds) and around them, against the oracle."""
import numpy as np
import pytest

from oracle import afqmc as O
from paper_2003_01831_gb300 import synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nu,Nd", [(1, 2), (8, 9), (31, 32), (33, 40), (64, 65), (100, 116), (117, 118), (127, 128)])
def test_local_energy_and_step(Nu, Nd):
    M, nch, W, tau = max(Nu, Nd) + 12, 7, 5, 0.005
    rng = np.random.default_rng(Nu)
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, Nu, Nd)
    Phi0 = [p[None] + 0.3 / np.sqrt(M) * (rng.standard_normal((W,) + p.shape) + 1j * rng.standard_normal((W,) + p.shape))
            for p in Psi]
    x = syn.make_fields(1, W, nch, seed=2)
    ham = O.Hamiltonian(h=h, L=L, E0=E0)
    wk = O.init_walkers(ham, Psi, W, Phi0)
    with AFQMC(h, L, E0, Psi[0], Psi[1], W, tau, Phi0=Phi0, k_qr=0) as g:
        E = g.energy()[0]
        ref = O.local_energy(ham, Psi, Phi0)[0]
        assert np.max(np.abs(E - ref)) < 1e-11 * np.max(np.abs(ref))
        g.step(1, x)
        w = g.energy()[1]
    O.step(ham, Psi, O.half_one_body_propagator(ham, tau), wk, x[0], O.Params(tau=tau))
    assert np.max(np.abs(w - wk.w)) < 1e-11 * np.max(wk.w)
