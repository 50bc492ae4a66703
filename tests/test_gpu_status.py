"""A bounded wait that gave up in a product of a gradient or of a walker set's set-up is reported by that call
(the status word is raised by hand: no wait runs out here)."""
import ctypes

import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu
TIMEOUT = 4


def set_status(wk, bits):
    lib = api.lib()
    lib.afqmc_debug_set_status.argtypes = [ctypes.c_void_p, ctypes.c_uint]
    assert lib.afqmc_debug_set_status(wk, bits) == 0


def system():
    h, L, E0 = syn.make_hamiltonian(12, 10, np.random.default_rng(2))
    Psi = syn.make_trial(h, 3, 3)
    return h, L, E0, Psi[0], Psi[1], 4, 0.01


def test_gradient_reports_a_timeout():
    d = np.ones(4, complex)
    with AFQMC(*system()) as g:
        g.backward(d, d)
        set_status(g.wk, TIMEOUT)
        with pytest.raises(api.AfqmcError, match="TIMEOUT"):
            g.backward(d, d)


def test_set_up_reports_a_timeout():
    set_status(None, TIMEOUT)
    try:
        with pytest.raises(api.AfqmcError, match="TIMEOUT"):
            AFQMC(*system())
    finally:
        set_status(None, 0)
    with AFQMC(*system()) as g:
        assert np.all(np.isfinite(g.energy()[0]))
