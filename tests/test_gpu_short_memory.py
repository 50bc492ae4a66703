"""Calls on an FP64 walker set that find no device memory at first: the set gives back the workspace of its
tensor-core products, the call goes on, and its results are those with the workspace to FP64 rounding."""
import ctypes

import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


def run(short, call, slices):
    """The results of a walker set's call; `short` of its allocations fail at first."""
    lib = api.lib()
    lib.afqmc_debug_short_allocs.argtypes = [ctypes.c_int]
    lib.afqmc_debug_slice_bytes.argtypes = [ctypes.c_void_p]
    lib.afqmc_debug_slice_bytes.restype = ctypes.c_longlong
    rng = np.random.default_rng(5)
    M, N, nch, W = 96, 24, 200, 64
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    x = rng.standard_normal((2, W, nch))
    try:
        lib.afqmc_debug_short_allocs(short if call == "set-up" else 0)
        with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, k_qr=2) as g:
            lib.afqmc_debug_short_allocs(short if call == "window" else 0)
            g.bp_begin(2)
            out = [g.step(2, x, measure_every=1)]
            lib.afqmc_debug_short_allocs(short if call == "estimate" else 0)
            out += g.bp_rdm1()
            lib.afqmc_debug_short_allocs(short if call == "gradient" else 0)
            out += g.backward(np.ones(W, complex), np.ones(W, complex))
            out += g.energy()[:3]
            slices.append(lib.afqmc_debug_slice_bytes(g.wk))
    finally:
        lib.afqmc_debug_short_allocs(0)
    return out


@pytest.mark.parametrize("call", ["set-up", "window", "estimate", "gradient"])
def test_room_is_given_back(call):
    slices = []
    want, got = run(0, call, slices), run(1, call, slices)
    assert slices[0] > 0 and slices[1] == 0
    for a, b in zip(got, want):
        assert np.max(np.abs(np.asarray(a) - np.asarray(b))) < 1e-11 * np.max(np.abs(b))
