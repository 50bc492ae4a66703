"""FP64 walker sets where device memory does not hold the whole workspace of the tensor-core products: a part of
it, or none, gives the same steps."""
import ctypes

import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


def test_any_room_will_do():
    lib = api.lib()
    lib.afqmc_debug_set_slice_room.argtypes = [ctypes.c_longlong]
    rng = np.random.default_rng(4)
    M, N, nch, W = 96, 24, 200, 64
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    x = rng.standard_normal((2, W, nch))
    runs = []
    try:
        for room in (-1, 30 << 20, 9 << 20, 1 << 20, 0):
            lib.afqmc_debug_set_slice_room(room)
            with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, k_qr=2) as g:
                trace = g.step(2, x, measure_every=1)
                runs.append([trace, *g.energy()[:3], *g.backward(np.ones(W, complex), np.ones(W, complex))])
    finally:
        lib.afqmc_debug_set_slice_room(-1)
    for r in runs[1:]:
        for got, want in zip(r, runs[0]):
            assert np.max(np.abs(got - want)) < 1e-11 * np.max(np.abs(want))
