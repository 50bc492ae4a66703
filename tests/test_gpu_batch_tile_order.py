"""Tiles of different electron counts one after another on the same CTAs of a batch's one energy launch:
N' = 64 and 128 before and after N' = 32, with Cholesky vectors that decay fast, so that most tiles
form the single product and their accumulators are ready before the tile before them is read out.
Every system has about one tile for each CTA pair, so a pair's consecutive tiles are of consecutive systems.
The arithmetic of a tile does not depend on its neighbours: repeats, and one launch per system, give
the same bits."""
import ctypes

import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import Batch

pytestmark = pytest.mark.gpu

A32 = (128, 32, 608, 2)    # (M, N, Nchol, W): 76 pair tiles each
A64 = (128, 64, 304, 1)
A128 = (192, 128, 76, 1)


@pytest.mark.parametrize("order", [(A64, A32), (A128, A32), (A32, A64, A32, A128, A32), (A64, A32, A64, A32, A64, A32)])
def test_tiles_of_other_sizes(order):
    systems = []
    for i, (M, N, nchol, W) in enumerate(order):
        h, L, E0, Psi = syn.make_uneven_system(syn.UnevenSystem(M=M, N=N, Nchol=nchol, W=W), i, seed=21, decay=3.0)
        systems.append((h, L, E0, Psi[0], Psi[1], W))
    lib = api.lib()
    lib.afqmc_debug_set_batch_energy.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    runs = []
    for multi in (0, 1, 1, 1):
        with Batch(systems, 0.005, precision=api.PREC_BF16X3) as b:
            assert lib.afqmc_debug_set_batch_energy(b.b, multi, 32) == 0
            trace = b.step(6, seed=5, measure_every=1)
            runs.append([trace] + [b.energy(s)[0] for s in range(len(order))])
    assert np.all(np.isfinite(runs[0][0]))
    for r in runs[1:]:
        for got, want in zip(r, runs[0]):
            assert np.array_equal(got, want)
