"""The three-slice products on CTA pairs (contractions of 512 and more, two or more row tiles): the
propagation of mixed walker sets at even and odd numbers of row tiles against the FP64 path."""
import numpy as np
import pytest

from paper_2003_01831_gb300 import api, synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,nch,W", [(64, 8, 512, 65), (64, 16, 576, 128), (64, 8, 520, 190), (64, 8, 512, 520), (64, 8, 512, 577),
                                       (256, 64, 512, 3), (256, 72, 64, 2)])
def test_step_follows_fp64(M, N, nch, W):
    rng = np.random.default_rng(M + N + nch + W)
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    x = rng.standard_normal((2, W, nch))
    out = {}
    for prec in (api.PREC_FP64, api.PREC_BF16X3):
        with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, precision=prec, k_qr=0) as g:
            g.step(2, x)
            out[prec] = g.walkers()[:3]
    for a, b in zip(out[api.PREC_BF16X3], out[api.PREC_FP64]):
        # three slices an operand (2^-30) in some twenty products a step, force biases of two slices (2^-21)
        assert np.max(np.abs(a - b)) < 1e-5 * np.max(np.abs(b))
