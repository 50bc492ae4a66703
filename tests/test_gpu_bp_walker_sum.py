"""The tensor-core walker sum of a back-propagated estimate (its operands packed and sliced a block or
a warp to a row) at contraction lengths 2 W N below, at and past 512, and past one chunk of 8192, with dead
walkers: a zero-length window is the mixed estimate sum_w w Theta_w Psi^+ / sum_w w."""
import numpy as np
import pytest

from oracle import backprop as BP
from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 31, 32, 33, 130, 512, 520])
def test_zero_length_window(W):
    rng = np.random.default_rng(W)
    M, N, nch = 64, 8, 64
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    Phi0 = [syn.make_random_walkers(M, N, W, 3 + s) + 2.0 * Psi[s][None] for s in range(2)]
    with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.01, Phi0=Phi0, precision=api.PREC_BF16X3) as g:
        Pu, Pd, w, step = g.walkers()
        w = rng.uniform(0.5, 1.5, W).astype(w.dtype)
        w[1::7] = 0.0
        g.set_walkers(Pu, Pd, w, step)
        g.bp_begin(0)
        G = g.bp_rdm1()
    ref = BP.Window([Pu, Pd]).estimate(L, Psi, np.eye(M), w, 0.01, 6)
    for s in range(2):
        # Theta from two fp16 slices an operand (2^-21 of its rows' norms), overlaps of condition ~10
        assert np.max(np.abs(G[s] - ref[s])) < 10 * 2.0 ** -21 * max(1.0, np.max(np.abs(ref[s])))
