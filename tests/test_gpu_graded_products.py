"""FP64 products on the tensor cores whose entries differ in size along the contraction: within rows at
random, large entries of the one operand against small ones of the other (walker columns of
different norms), one side decaying, imaginary parts far below the real ones, numbers near the ends of
the FP64 range.  Against long double sums: every component within the bound of the multiply-add
loop, and in the norm no further off than that loop."""
import numpy as np
import pytest

from paper_2003_01831_gb300 import synthetic as syn
from paper_2003_01831_gb300.walkers import AFQMC
from test_gpu_gemm_slices import C_, N_, T_, gemm, long_product, op_of, rand

pytestmark = pytest.mark.gpu


def both(A, B, m, n, k, ar=0, br=0, opa=N_, opb=N_, **kw):
    kw = dict(a=(ar, opa, A.shape[1], (0, 0, 0)), b=(br, opb, B.shape[1], (0, 0, 0)), ldc=n, **kw)
    C = np.full((m, n), np.nan + 0j)
    return gemm(A, B, C, m, n, k, **kw)[0], gemm(A, B, C, m, n, k, form=0, **kw)[0]


def check(got, old, A, B, norm=True):
    re, im = long_product(A, B)
    a, b = ([np.abs(np.asarray(f(X), float)) for f in (np.real, np.imag)] for X in (A, B))
    sizes = a[0] @ b[0] + a[1] @ b[1], a[0] @ b[1] + a[1] @ b[0]
    k = (1 + np.iscomplexobj(A)) * A.shape[-1] if np.iscomplexobj(A) == np.iscomplexobj(B) else A.shape[-1]
    new = [np.asarray(g - e, float) for g, e in zip((got.real, got.imag), (re, im))]
    was = [np.asarray(g - e, float) for g, e in zip((old.real, old.imag), (re, im))]
    for err, size in zip(new, sizes):   # k roundings of the loop, or the digits' part of them; 2^-1070: subnormal results
        assert np.all(np.abs(err) <= (k + 2) * 2.0 ** -53 * size + 2.0 ** -1070)
    for err, before, size in zip(new, was, sizes) if norm else ():
        s = np.where(size > 0, size, 1.0)
        assert np.linalg.norm(err / s) <= np.linalg.norm(before / s) * (1 + 1e-12)


def grade(rng, decades, k):
    return 10.0 ** rng.uniform(0, decades, k) if decades else np.ones(k)


@pytest.mark.parametrize("ar,br", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("decades", [0, 1, 2, 4, 8, 16])
@pytest.mark.parametrize("m,n,k", [(64, 50, 16), (130, 33, 64), (40, 70, 128), (33, 260, 129), (50, 40, 300)])
def test_opposite_grades(ar, br, decades, m, n, k):
    rng = np.random.default_rng(decades * 1000 + k + 2 * ar + br)
    s = grade(rng, decades, k)
    A, B = rand(rng, ar, m, k) * s, rand(rng, br, k, n) / s[:, None]
    check(*both(A, B, m, n, k, ar, br), A, B)


@pytest.mark.parametrize("opa,opb", [(N_, T_), (C_, N_), (T_, C_)])
@pytest.mark.parametrize("k", [24, 96, 200])
def test_ranges_within_rows(opa, opb, k):
    rng = np.random.default_rng(k + 10 * opa + opb)
    m, n = 70, 90
    for la, lb in ((40, 0), (0, 40), (20, 20), (60, 60)):
        A = rand(rng, 0, *((m, k) if opa == N_ else (k, m)))
        B = rand(rng, 0, *((k, n) if opb == N_ else (n, k)))
        A = A * np.exp2(rng.integers(-la, 1, A.shape).astype(float))
        B = B * np.exp2(rng.integers(-lb, 1, B.shape).astype(float))
        check(*both(A, B, m, n, k, opa=opa, opb=opb), op_of(A, opa), op_of(B, opb))


def test_decay_small_imaginary_parts_and_disjoint_rows():
    rng = np.random.default_rng(3)
    m, n, k = 90, 80, 384
    d = np.exp(-np.arange(k) / 20.0)
    A, B = rand(rng, 0, m, k), rand(rng, 1, k, n) * d[:, None]
    check(*both(A, B, m, n, k, 0, 1), A, B)
    A = A * d
    check(*both(A, B, m, n, k, 0, 1), A, B)
    A, B = A.real + 1e-9j * A.imag, rand(rng, 0, k, n).real + 1e-7j * rand(rng, 1, k, n)
    check(*both(A, B, m, n, k), A, B)
    A, B = rand(rng, 0, m, k), rand(rng, 0, k, n)
    A[::2, ::2] = 0.0
    B[1::2, ::2] = 0.0       # rows 0, 2, ... of A meet zeros in the even columns of B
    got, old = both(A, B, m, n, k)
    check(got, old, A, B)
    assert np.all(got[::2, ::2] == 0)


@pytest.mark.parametrize("k", [48, 96])
def test_ends_of_the_range(k):
    """Infinities and NaN, subnormal numbers, products beyond the range: as the loop gives."""
    rng = np.random.default_rng(4)
    m, n = 60, 70
    A, B = rand(rng, 0, m, k), rand(rng, 0, k, n)
    A[1], A[2], A[3] = A[1] * 1e-305, A[2] * 1e300, 0.0
    B[:, 1], B[:, 2], B[:, 3] = B[:, 1] * 1e-300, B[:, 2] * 1e300, 0.0
    A[4, 7], A[5, 0], B[9, 4], A[6, 5], B[5, 6] = np.inf, np.nan, -np.inf, 1e308, 1e308
    A[7] = A[7].real
    A[8] = 1e-310 * A[8]
    got, old = both(A, B, m, n, k)
    # (whether sums of infinities end as one or as NaN depends on their order)
    assert np.array_equal(np.isfinite(got), np.isfinite(old))
    rows, cols = [i for i in range(m) if i not in (2, 4, 5, 6)], [j for j in range(n) if j not in (2, 4, 6)]
    check(got[np.ix_(rows, cols)], old[np.ix_(rows, cols)], A[rows], B[:, cols])
    assert np.all(got[3, :4] == 0) and np.all(got[:4, 3] == 0)


@pytest.mark.parametrize("k", [16, 100, 128, 300])
def test_equal_entries_of_the_largest_digits(k):
    """Every digit at the end of its range and every product of one sign: the accumulators' largest values."""
    m, n = 70, 90
    for lead in (64, 100, 127):
        v = lead * 2 ** 51 + 128 * (2 ** 43 + 2 ** 35 + 2 ** 27 + 2 ** 19)
        x = -v * 2.0 ** -58
        for A, B in ((np.full((m, k), x), np.full((k, n), x)), (np.full((m, k), x), np.full((k, n), -x)),
                     (np.full((m, k), x * (1 + 1j)), np.full((k, n), x * (1 - 1j)))):
            cplx = int(not np.iscomplexobj(A))
            check(*both(A, B, m, n, k, cplx, cplx), A, B, norm=False)   # one value: its error is no statistic


def test_alpha_beta_second_output_of_looped_results():
    rng = np.random.default_rng(6)
    m, n, k, W = 50, 70, 200, 3
    s = grade(rng, 12, k)
    A, B, C, D = rand(rng, 0, W, m, k) * s, rand(rng, 0, k, n) / s[:, None], rand(rng, 0, W, m, n), rand(rng, 0, W, m, n + 3)
    kw = dict(nb=(1, W, 1), a=(0, N_, k, (0, m * k, 0)), b=(0, N_, n, (0, 0, 0)), ldc=n, sc=(0, m * n, 0), ldd=n + 3,
              sd=(0, m * (n + 3), 0))
    for alpha, beta in ((-1.0, 1.0), (0.25j, 0.0), (0.3 - 0.7j, 0.5)):
        got, Dg, _, _ = gemm(A, B, C, m, n, k, alpha=alpha, beta=beta, D=D, **kw)
        ref, Dr, _, _ = gemm(A, B, C, m, n, k, alpha=alpha, beta=beta, D=D, form=0, **kw)
        tol = 4 * k * 2.0 ** -52 * (np.max(np.abs(A) @ np.abs(B)) + 4)
        assert np.max(np.abs(got - ref)) < tol and np.max(np.abs(Dg - Dr)) < tol
        assert np.array_equal(Dg[..., n:], D[..., n:])


def test_walkers_of_unequal_column_norms():
    """Columns scaled by powers of two leave E_L as it is, to the bit in the multiply-add form."""
    rng = np.random.default_rng(7)
    M, N, nch, W = 96, 24, 200, 48
    h, L, E0 = syn.make_hamiltonian(M, nch, rng)
    Psi = syn.make_trial(h, N, N)
    F = Psi[0][None] + 0.05 * (rng.standard_normal((W, M, N)) + 1j * rng.standard_normal((W, M, N)))
    E = []
    for spread in (0, 30):
        s = np.exp2(rng.integers(-spread, 1, (W, 1, N)).astype(float))
        with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.005, Phi0=(F * s, F * s)) as g:
            E.append(g.energy()[0])
    assert np.max(np.abs(E[1] - E[0])) < 1e-13 * np.max(np.abs(E[0]))


@pytest.mark.parametrize("cplx", [False, True])
def test_step_at_sizes_of_the_tensor_core_form(cplx):
    """One-body propagator (its diagonal apart), Taylor terms and energy against the oracle."""
    import test_gpu_complex_cholesky as C
    import test_gpu_fp64 as F
    M, N, W = 72, 18, 40
    if cplx:
        h, L, Psi, rng = C.complex_system(M, N, N, 40, seed=8, scale=0.3)
        x = rng.standard_normal((2, W, 80))
        C.run_parity(h, L, 0.1, Psi, W, 0.005, 2, 2, x)
    else:
        rng = np.random.default_rng(9)
        h, L, E0 = syn.make_hamiltonian(M, 144, rng)
        x = rng.standard_normal((2, W, 144))
        F.run_parity(h, L, E0, syn.make_trial(h, N, N), W, 0.005, 2, 2, x)


def test_gradients_at_sizes_of_the_tensor_core_form():
    """The terms of Theta T_n and of c_n Theta, formed apart."""
    import test_gpu_backward as B
    from oracle import afqmc as O
    M, N, nch, W = 72, 18, 144, 40
    h, L, E0, Psi, Phi, dE, dS = B.instance(M, N, nch, W, 12)
    with AFQMC(h, L, E0, Psi[0], Psi[1], W, 0.01, Phi0=Phi) as g:
        got = g.backward(dE, dS)
    for a, b in zip(got, B.energy_logdet_backward(O.Hamiltonian(h, L, E0), Psi, Phi, dE, dS)):
        assert B.rel(a, b) < 1e-10
