"""The tensor-core form of the FP64 products (operands sliced into exact fp16 digits) against long
double sums and against the multiply-add kernel it replaces: every operand form (real or complex, N,
T or C), batch dimensions of either operand and shared, sizes at the edges of tiles, stages and
digit widths, alpha, beta and the second output, workspaces too small for the whole product, and rows with
infinities or wide ranges."""
import ctypes
import itertools

import numpy as np
import pytest

from paper_2003_01831_gb300 import api

pytestmark = pytest.mark.gpu
N_, T_, C_ = 0, 1, 2


def gemm(A, B, C, m, n, k, nb=(1, 1, 1), a=(0, N_, 0, (0, 0, 0)), b=(0, N_, 0, (0, 0, 0)), ldc=0, sc=(0, 0, 0),
         alpha=1.0, beta=0.0, D=None, ldd=0, sd=(0, 0, 0), form=1, ws=256 << 20, reps=0):
    L = api.lib()
    vp = ctypes.c_void_p
    L.afqmc_debug_gemm.restype = ctypes.c_int
    L.afqmc_debug_gemm.argtypes = [vp, vp, vp, vp, vp, vp, vp, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, vp, vp]
    d = np.array([m, n, k, *nb, a[0], a[1], a[2], *a[3], b[0], b[1], b[2], *b[3], ldc, *sc, ldd, *sd, 0, 0], dtype=np.int64)
    sizes = np.array([A.size, B.size, C.size, 0 if D is None else D.size], dtype=np.int64)
    ab = np.array([complex(alpha).real, complex(alpha).imag, complex(beta).real, complex(beta).imag])
    C = C.copy()
    Dc = None if D is None else D.copy()
    chose, ms = ctypes.c_int(), ctypes.c_float()
    rc = L.afqmc_debug_gemm(d.ctypes.data, sizes.ctypes.data, ab.ctypes.data, A.ctypes.data, B.ctypes.data, C.ctypes.data,
                            None if Dc is None else Dc.ctypes.data, form, ws, reps, ctypes.addressof(chose),
                            ctypes.addressof(ms))
    assert rc == 0, api.afqmc_last_error()
    return C, Dc, chose.value, ms.value


def rand(rng, real, *shape):
    x = rng.standard_normal(shape)
    return x if real else x + 1j * rng.standard_normal(shape)


def op_of(X, op):
    return X if op == N_ else (np.swapaxes(X, -1, -2) if op == T_ else np.conj(np.swapaxes(X, -1, -2)))


def long_product(A, B):
    """A B in long double (complex by parts), over leading batch dimensions."""
    ar, ai = (np.asarray(f(A), dtype=np.longdouble) for f in (np.real, np.imag))
    br, bi = (np.asarray(f(B), dtype=np.longdouble) for f in (np.real, np.imag))
    return ar @ br - ai @ bi, ar @ bi + ai @ br


def check(got, A, B, other=None, scale=1.0):
    re, im = long_product(A, B)
    err = np.hypot(np.asarray(got.real - re, dtype=float), np.asarray(got.imag - im, dtype=float))
    na = np.linalg.norm(A, axis=-1)[..., :, None]
    nb = np.linalg.norm(B, axis=-2)[..., None, :]
    size = np.hypot(np.asarray(re, dtype=float), np.asarray(im, dtype=float))
    # operands rounded 2^-58 below their largest entry, dropped weights 2^-56 below the largest
    # products (random signs), one rounding of the result
    assert np.all(err <= 2.0 ** -50 * scale * na * nb + 2.0 ** -52 * size), np.max(err / (na * nb + 1e-300))
    if other is not None:
        old = np.hypot(np.asarray(other.real - re, dtype=float), np.asarray(other.imag - im, dtype=float))
        assert np.linalg.norm(err) <= np.linalg.norm(old), (np.linalg.norm(err), np.linalg.norm(old))


@pytest.mark.parametrize("ar,br", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (5, 7, 3), (64, 128, 32), (65, 129, 33), (63, 127, 64), (32, 32, 65),
                                   (130, 70, 128), (33, 40, 129), (40, 33, 256), (20, 50, 300), (17, 9, 700)])
def test_forms_and_edges(ar, br, m, n, k):
    rng = np.random.default_rng(m * 1000 + n + k)
    for opa, opb in itertools.product((N_, T_, C_), repeat=2):
        if (opa == C_ and ar) or (opb == C_ and br) or (m > 60 and (opa, opb) not in ((N_, N_), (C_, N_), (T_, T_))):
            continue
        A = rand(rng, ar, m, k) if opa == N_ else rand(rng, ar, k, m)
        B = rand(rng, br, k, n) if opb == N_ else rand(rng, br, n, k)
        kw = dict(a=(ar, opa, A.shape[1], (0, 0, 0)), b=(br, opb, B.shape[1], (0, 0, 0)), ldc=n)
        C = np.full((m, n), np.nan + 0j)
        got = gemm(A, B, C, m, n, k, **kw)[0]
        old = gemm(A, B, C, m, n, k, form=0, **kw)[0]
        check(got, op_of(A, opa), op_of(B, opb), old if k >= 32 and m * n >= 1000 else None)
        # one output per thread: the same sums in the same order as the tiles
        assert np.array_equal(gemm(A, B, C, m, n, k, form=3, **kw)[0], old)


@pytest.mark.parametrize("ws", [256 << 20, 300 << 10])
def test_batches(ws):
    """Batch dimensions of either operand and shared, also in a workspace too small for the whole
    product.  The shapes of the step: Psi^+ Phi_w, Ltilde_n Theta_w over (n, w), Phi_w S_w^-1, three batch
    dimensions, and outputs in a transposed batch order."""
    rng = np.random.default_rng(1)
    M, N, W, nc, nd = 37, 9, 7, 5, 3
    Psi, Phi = rand(rng, 0, M, N), rand(rng, 0, W, M, N)
    got = gemm(Psi, Phi, np.zeros((W, N, N), complex), N, N, M, nb=(1, W, 1), a=(0, C_, N, (0, 0, 0)),
               b=(0, N_, N, (0, M * N, 0)), ldc=N, sc=(0, N * N, 0), ws=ws)[0]
    check(got, np.broadcast_to(Psi.conj().T, (W, N, M)), Phi)
    for real in (0, 1):
        Lt = rand(rng, real, nc, N, M)
        got = gemm(Lt, Phi, np.zeros((nc, W, N, N), complex), N, N, M, nb=(1, nc, W), a=(real, N_, M, (0, N * M, 0)),
                   b=(0, N_, N, (0, 0, M * N)), ldc=N, sc=(0, W * N * N, N * N), ws=ws)[0]
        check(got, np.broadcast_to(Lt[:, None], (nc, W, N, M)), np.broadcast_to(Phi[None], (nc, W, M, N)))
    Si = rand(rng, 0, W, N, N)
    got = gemm(Phi, Si, np.zeros((W, M, N), complex), M, N, N, nb=(1, W, 1), a=(0, N_, N, (0, M * N, 0)),
               b=(0, N_, N, (0, N * N, 0)), ldc=N, sc=(0, M * N, 0), ws=ws)[0]
    check(got, Phi, Si)
    LtI, ThI = rand(rng, 0, nd, nc, N, M), rand(rng, 0, nd, W, M, N)
    got = gemm(LtI, ThI, np.zeros((nc, nd, W, N, N), complex), N, N, M, nb=(nc, nd, W),
               a=(0, N_, M, (N * M, nc * N * M, 0)), b=(0, N_, N, (0, W * M * N, M * N)), ldc=N,
               sc=(nd * W * N * N, W * N * N, N * N), ws=ws)[0]
    A = np.broadcast_to(np.moveaxis(LtI, 1, 0)[:, :, None], (nc, nd, W, N, M))
    check(got, A, np.broadcast_to(ThI[None], (nc, nd, W, M, N)))
    # U[w][c] = Theta_w T[c][w]: the output's batch order differs from B's
    T = rand(rng, 0, nc, W, N, N)
    got = gemm(Phi, T, np.zeros((W, nc, M, N), complex), M, N, N, nb=(1, W, nc), a=(0, N_, N, (0, M * N, 0)),
               b=(0, N_, N, (0, N * N, W * N * N)), ldc=N, sc=(0, nc * M * N, M * N), ws=ws)[0]
    check(got, np.broadcast_to(Phi[:, None], (W, nc, M, N)), np.moveaxis(T, 1, 0))


@pytest.mark.parametrize("ar,br", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_alpha_beta_and_second_output(ar, br):
    rng = np.random.default_rng(5)
    m, n, k = 50, 70, 600
    A, B, C, D = rand(rng, ar, m, k), rand(rng, br, k, n), rand(rng, 0, m, n), rand(rng, 0, m, n + 3)
    kw = dict(a=(ar, N_, k, (0, 0, 0)), b=(br, N_, n, (0, 0, 0)), ldc=n, ldd=n + 3)
    for alpha, beta in ((-1.0, 1.0), (0.25j, 0.0), (0.3 - 0.7j, 0.5), (2.0, 1.0)):
        if ar and br and complex(alpha).imag != 0:
            continue
        got, Dg, _, _ = gemm(A, B, C, m, n, k, alpha=alpha, beta=beta, D=D, **kw)
        ref, Dr, _, _ = gemm(A, B, C, m, n, k, alpha=alpha, beta=beta, D=D, form=0, **kw)
        tol = 1e-15 * 40 * k ** 0.5 * 4
        assert np.max(np.abs(got - ref)) < tol and np.max(np.abs(Dg - Dr)) < tol
        assert np.array_equal(Dg[:, n:], D[:, n:])


@pytest.mark.parametrize("ar,br,ws", [(0, 0, 256 << 20), (0, 0, 2 << 20), (1, 0, 256 << 20), (0, 1, 3 << 20)])
def test_long_contractions(ar, br, ws):
    """Few output tiles and a long contraction: its pieces are shared between CTAs, and between rounds
    where the workspace is small."""
    rng = np.random.default_rng(6)
    m, n, k, W = 40, 12, 5003, 3
    A, B, C = rand(rng, ar, m, k), rand(rng, br, W, k, n), rand(rng, 0, W, m, n)
    got, D, _, _ = gemm(A, B, C, m, n, k, nb=(1, W, 1), a=(ar, N_, k, (0, 0, 0)), b=(br, N_, n, (0, k * n, 0)), ldc=n,
                        sc=(0, m * n, 0), beta=1.0, D=C, ldd=n, sd=(0, m * n, 0), ws=ws)
    re, im = long_product(np.broadcast_to(A, (W, m, k)), B)
    tol = 2.0 ** -50 * np.linalg.norm(A, axis=-1)[:, None] * np.linalg.norm(B, axis=-2)[:, None, :]
    assert np.all(np.hypot(np.asarray(got.real - re - C.real, float), np.asarray(got.imag - im - C.imag, float)) < tol)
    assert np.max(np.abs(D - C - got)) < 1e-12


def test_ranges_and_special_values():
    rng = np.random.default_rng(9)
    m, n, k = 40, 130, 96
    A = rand(rng, 0, m, k) * np.exp2(rng.integers(-300, 300, (m, 1)).astype(float))   # rows far apart
    B = rand(rng, 0, k, n) * np.exp2(rng.integers(-200, 200, (1, n)).astype(float))
    kw = dict(a=(0, N_, k, (0, 0, 0)), b=(0, N_, n, (0, 0, 0)), ldc=n)
    check(gemm(A, B, np.zeros((m, n), complex), m, n, k, **kw)[0], A, B)
    A = rand(rng, 0, m, k) * np.exp2(rng.integers(-40, 1, (m, k)).astype(float))      # and within rows
    check(gemm(A, B, np.zeros((m, n), complex), m, n, k, **kw)[0], A, B)
    A[3] = 0.0
    B[:, 5] = 0.0
    A[7, 2], A[9, 0], B[4, 11] = np.inf, np.nan, -np.inf
    got = gemm(A, B, np.zeros((m, n), complex), m, n, k, **kw)[0]
    bad = np.zeros((m, n), bool)
    bad[[7, 9]] = bad[:, 11] = True
    assert np.all(~np.isfinite(got[bad])) and np.all(np.isfinite(got[~bad]))
    assert np.all(got[3][~bad[3]] == 0) and np.all(got[~bad[:, 5], 5] == 0)
    # results beyond the FP64 range
    A, B = np.full((m, k), 1e200), np.full((k, n), 1e200)
    kw = dict(a=(1, N_, k, (0, 0, 0)), b=(1, N_, n, (0, 0, 0)), ldc=n)
    assert np.all(np.isinf(gemm(A, B, np.zeros((m, n), complex), m, n, k, **kw)[0].real))
    assert np.all(gemm(1 / A, 1 / B, np.zeros((m, n), complex), m, n, k, **kw)[0] == 0)
