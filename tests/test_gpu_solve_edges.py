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
