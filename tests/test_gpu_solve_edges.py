"""The generalized eigenproblem on pencils that have no solution: a NaN or an infinity in the triangle that is used
is an error, whatever the size, and never energies."""
import numpy as np
import pytest

from paper_2404_10223_gb300 import tnqe

pytestmark = pytest.mark.gpu
NOCONV = 5


@pytest.fixture(scope="module")
def ctx():
    import os
    from paper_2404_10223_gb300 import build as B
    if not os.path.exists(B.LIB):
        B.build()
    with tnqe.Context(np.zeros((2, 2)), np.zeros((2, 2, 2, 2)), 2, 1, 1) as g:
        yield g


def pencil(M, seed=0):
    rng = np.random.default_rng([M, seed])
    A = rng.normal(size=(M, M))
    Y = rng.normal(size=(M, M + 4)) / np.sqrt(M)
    return A + A.T - 20.0 * np.diag(np.arange(M)), np.eye(M) + Y @ Y.T


@pytest.mark.parametrize("M", [1, 2, 3, 32])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("which", ["H", "S", "S of the identity"])
def test_entry_that_is_not_finite_is_an_error(ctx, M, bad, which):
    for i, j in {(0, 0), (0, M - 1), (M // 2, M - 1), (M - 1, M - 1)}:
        H, S = pencil(M)
        if which == "S of the identity":
            S = np.eye(M)
        (H if which == "H" else S)[i, j] = bad
        with pytest.raises(tnqe.TnqeError) as e:
            ctx.solve(H, S)
        assert e.value.status == NOCONV
        if which != "H" and j < M - 1:                # rows 0..M-2 enter an eigenproblem of the residuals
            with pytest.raises(tnqe.TnqeError) as e:
                ctx.dependence(S)
            assert e.value.status == NOCONV


@pytest.mark.parametrize("M", [2, 3, 32])
def test_the_lower_triangle_is_not_read(ctx, M):
    H, S = pencil(M)
    ref = ctx.solve(H, S)
    Hl, Sl = H.copy(), S.copy()
    Hl[M - 1, 0] = np.nan
    Sl[M - 1, 0] = np.inf
    got = ctx.solve(Hl, Sl)
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1]) and ref[2:] == got[2:]


@pytest.mark.parametrize("M", [2, 3, 28])
@pytest.mark.parametrize("e", [-900, -300, 300, 1014])
def test_pencils_near_the_ends_of_the_exponent_range(ctx, M, e):
    """H times a power of two: the energies times the same, exactly (the norm of H for M = 28 is above 2^9)."""
    H, S = pencil(M)
    E, C, r, _ = ctx.solve(H, S)
    E2, C2, r2, _ = ctx.solve(np.ldexp(H, e), S)
    assert r == r2 == M and np.array_equal(np.ldexp(E, e), E2) and np.array_equal(C, C2)


@pytest.mark.parametrize("M", [2, 3, 4, 5, 8, 24, 32])
@pytest.mark.parametrize("span", [0, 4, 10, 22])
def test_graded_pencils_keep_the_relative_accuracy_of_jacobi(ctx, M, span):
    """D H D and D S D with D from 1 down to 10^-span: the same energies.  Jacobi's method resolves the small eigenvalues
    of S relative to themselves (Demmel and Veselic, SIAM J. Matrix Anal. Appl. 13 (1992) 1204)."""
    for seed in range(3):
        H, S = pencil(M, seed)
        L = np.linalg.cholesky(S)
        ref = np.linalg.eigvalsh(np.linalg.solve(L, np.linalg.solve(L, H).T))
        D = np.ldexp(1.0, -np.round(span * np.log2(10.0) * np.arange(M) / M).astype(int))   # powers of two: exact
        E, C, r, _ = ctx.solve_ex(H * D[:, None] * D, S * D[:, None] * D, 0.0)
        assert r == M
        # rounding of either route: a few eps of the norms over the smallest eigenvalue of S (1)
        assert np.abs(E - ref).max() <= 64 * 2.2e-16 * M * np.abs(H).sum(0).max()
        Cs = C * D[:, None]
        assert np.abs(Cs.T @ S @ Cs - np.eye(M)).max() <= 64 * 2.2e-16 * M * np.abs(S).sum(0).max()
