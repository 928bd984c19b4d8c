"""The truncated block SVD of a gate at the sizes and spectra where its parts can go wrong.

tnqe_apply_gate_noalloc with the identity gate truncates a two-site tensor whose
charge blocks and singular values the test chooses: block sizes around the limits of
one, two, four and sixteen warps, spectra with a decay down to the cutoff, exact
degeneracy, rank deficiency, and bonds whose blocks do not fit the scratch.  The
reference is NumPy's SVD of the same matrix in FP64.
"""
import numpy as np
import pytest

from paper_2404_10223_gb300 import inputs, tnqe

pytestmark = pytest.mark.gpu
U48 = 2.0 ** -48                                  # double-float products of the SVD path


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    from paper_2404_10223_gb300 import build as B
    if not os.path.exists(B.LIB):
        B.build()
    tnqe.load()


def gate(A, B, qL, qM, qR, side, chi_max, cutoff, c=1.0, s=0.0):
    import torch
    dA, dB = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B))
    chl, chm, chr_ = A.shape[0], A.shape[2], B.shape[2]
    Ao = torch.zeros(chl * 4 * chi_max, dtype=torch.float64, device="cuda")
    Bo = torch.zeros(chi_max * 4 * chr_, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    k, q, disc = tnqe.tnqe_apply_gate_noalloc(dA.data_ptr(), dB.data_ptr(), chl, chm, chr_, qL, qM, qR, c, s, side,
                                              chi_max, cutoff, 60, Ao.data_ptr(), Bo.data_ptr(), 0)
    return (Ao[: chl * 4 * k].cpu().numpy().reshape(chl, 4, k), Bo[: k * 4 * chr_].cpu().numpy().reshape(k, 4, chr_),
            k, disc)


def one_block(rows, cols, sigma, rng):
    """A two-site tensor with one rows x cols block (local states 3, 3) of the given singular values."""
    r = len(sigma)
    u = np.linalg.qr(rng.normal(size=(rows, r)))[0]
    v = np.linalg.qr(rng.normal(size=(cols, r)))[0]
    A, B = np.zeros((rows, 4, r)), np.zeros((r, 4, cols))
    A[:, 3, :] = u
    B[:, 3, :] = sigma[:, None] * v.T
    return A, B, [17] * rows, [34] * r, [51] * cols


def check(A, B, An, Bn, k, disc, side, keep, cutoff, gap):
    th = np.tensordot(A, B, axes=([2], [0]))
    m = th.reshape(th.shape[0] * 4, -1)
    u, sg, vt = np.linalg.svd(m, full_matrices=False)
    kref = max(1, min(keep, int((sg > cutoff * sg[0]).sum())))
    assert k == kref
    # backward error of the products over the gap at the cut (the largest of the block: 1)
    tol = 4.0 * U48 * np.sqrt(m.size) / gap
    new = np.tensordot(An, Bn, axes=([2], [0])).reshape(m.shape)
    assert np.abs(new - (u[:, :k] * sg[:k]) @ vt[:k]).max() <= tol * sg[0]
    iso = Bn.reshape(k, -1) if side == 0 else An.reshape(-1, k).T
    # corrections stop at 1e-8, and their FP32 arithmetic leaves 1e-6 of them
    assert np.abs(iso @ iso.T - np.eye(k)).max() <= 2e-12
    ref = float((sg[k:] ** 2).sum())
    assert abs(disc - ref) <= 1e-10 * ref + 1e-13 * float((sg ** 2).sum()) * (k < len(sg))


# limits: one warp / two / four warps at 16 and 50, both arrays of four warps at 74, one at 104, the whole CTA
@pytest.mark.parametrize("rows,cols", [(1, 1), (2, 1), (5, 3), (8, 16), (15, 15), (16, 17), (17, 16), (31, 33), (49, 60),
                                       (50, 50), (66, 64), (74, 75), (75, 77), (104, 105), (106, 105), (128, 128),
                                       (128, 9), (3, 127)])
@pytest.mark.parametrize("side", [0, 1])
def test_linear_spectrum_truncated_to_a_third(rows, cols, side):
    rng = np.random.default_rng(rows * 1000 + cols + side)
    n = min(rows, cols)
    A, B, qL, qM, qR = one_block(rows, cols, 1.0 - 0.9 * np.arange(n) / n, rng)
    keep = max(1, n // 3)
    An, Bn, k, disc = gate(A, B, qL, qM, qR, side, keep, 1e-14)
    check(A, B, An, Bn, k, disc, side, keep, 1e-14, 0.9 / n)


@pytest.mark.parametrize("n", [4, 24, 60, 90])
def test_decay_to_the_cutoff_keeps_what_is_above_it(n):
    rng = np.random.default_rng(n)
    sg = 10.0 ** (-12.0 * np.arange(n) / n)
    A, B, qL, qM, qR = one_block(n + 3, n, sg, rng)
    An, Bn, k, disc = gate(A, B, qL, qM, qR, 0, n, 1e-7)
    th = np.tensordot(A, B, axes=([2], [0])).reshape((n + 3) * 4, -1)
    new = np.tensordot(An, Bn, axes=([2], [0])).reshape(th.shape)
    ref = np.linalg.svd(th, compute_uv=False)
    # a singular value equal to the cutoff up to rounding (n = 60 has one) may go either way
    assert int((ref > (1e-7 + 4.0 * U48) * ref[0]).sum()) <= k <= int((ref > (1e-7 - 4.0 * U48) * ref[0]).sum())
    # what is dropped is below the cutoff
    assert np.linalg.norm(new - th) <= 1.01 * np.linalg.norm(ref[k:]) + 4.0 * U48 * np.sqrt(th.size)
    assert np.abs(Bn.reshape(k, -1) @ Bn.reshape(k, -1).T - np.eye(k)).max() <= 2e-12


@pytest.mark.parametrize("n", [2, 4, 5, 8, 9])
@pytest.mark.parametrize("low", [1e-13, 1e-17, 1e-20, 1e-40])
def test_columns_of_very_different_lengths_converge(n, low):
    """Columns from 1 down to far below the rounding of the longest (their order and signs mixed), as a product of
    decaying bonds leaves them: the SVD ends and keeps what is above the cutoff."""
    rng = np.random.default_rng(n)
    d = 10.0 ** np.linspace(0.0, np.log10(low), n)[rng.permutation(n)]
    A, B, qL, qM, qR = one_block(n + 2, n, np.ones(n), rng)
    A[:, 3, :] = rng.normal(size=(n + 2, n)) * d
    B[:, 3, :] = np.eye(n)
    An, Bn, k, disc = gate(A, B, qL, qM, qR, 0, n, 1e-14)
    m = A[:, 3, :]
    new = np.tensordot(An, Bn, axes=([2], [0]))[:, 3, 3, :]
    # backward stable in the 2-norm: m n eps of the largest, plus what the cutoff drops
    assert np.linalg.norm(new - m) <= (4.0 * U48 * n + 1e-14 * n) * np.linalg.norm(m)
    assert np.abs(Bn.reshape(k, -1) @ Bn.reshape(k, -1).T - np.eye(k)).max() <= 2e-12


@pytest.mark.parametrize("n", [12, 30, 60, 90])
@pytest.mark.parametrize("close", [1e-3, 1e-6, 1e-9, 1e-12])
def test_close_singular_values_at_the_cut_keep_the_vectors_orthonormal(n, close):
    """Eight singular values within `close` of one another around the cut, down to where the approximate vectors mix
    kept and dropped ones and the refinement gives up."""
    rng = np.random.default_rng(n)
    k = n // 2
    sg = np.linspace(1.0, 0.05, n)
    sg[k - 4: k + 4] = sg[k] * (1.0 + close * np.linspace(1.0, -1.0, 8))
    A, B, qL, qM, qR = one_block(n + 1, n, sg, rng)
    An, Bn, kn, disc = gate(A, B, qL, qM, qR, 0, k, 1e-12)
    th = np.tensordot(A, B, axes=([2], [0])).reshape((n + 1) * 4, -1)
    new = np.tensordot(An, Bn, axes=([2], [0])).reshape(th.shape)
    assert kn == k
    # double-float vectors and products (sums of n terms)
    V = Bn.reshape(k, -1)
    assert np.abs(V @ V.T - np.eye(k)).max() <= 4.0 * U48 * np.sqrt(n)
    assert np.abs(th @ V.T - An.reshape(-1, k)).max() <= 4.0 * U48 * np.sqrt(n)
    # any k-dimensional choice among the close ones drops the same weight up to close^2 of it
    best = float((sg[k:] ** 2).sum())
    assert np.linalg.norm(new - th) ** 2 <= best * (1.0 + 1e-10 + 8.0 * close) and disc <= best * (1.0 + 1e-10 + 8.0 * close)


@pytest.mark.parametrize("n,rank", [(6, 6), (20, 20), (40, 17), (64, 30), (64, 64)])
def test_degenerate_and_rank_deficient_blocks_are_kept_whole(n, rank):
    rng = np.random.default_rng(n + rank)
    sg = np.ones(rank)
    A, B, qL, qM, qR = one_block(n, n + 2, sg, rng)
    An, Bn, k, disc = gate(A, B, qL, qM, qR, 1, 128, 1e-10)
    th = np.tensordot(A, B, axes=([2], [0]))
    assert k == rank and disc <= 1e-20
    assert np.abs(np.tensordot(An, Bn, axes=([2], [0])) - th).max() <= 4.0 * U48 * np.sqrt(th.size)
    assert np.abs(An.reshape(-1, k).T @ An.reshape(-1, k) - np.eye(k)).max() <= 2e-12


def test_blocks_beyond_the_scratch_take_the_serial_path():
    """chi = 128, one charge on each outer bond: four 128 x 128 blocks."""
    rng = np.random.default_rng(5)
    qM = sorted([17, 18, 33, 34] * 32)
    A, B = np.zeros((128, 4, 128)), np.zeros((128, 4, 128))
    ql, qr = [17] * 128, [34] * 128
    for j, q in enumerate(qM):
        for k in range(4):
            if 17 + (k & 1) * 16 + (k >> 1) == q:
                A[:, k, j] = rng.normal(size=128)
            if q + (k & 1) * 16 + (k >> 1) == 34:
                B[j, k, :] = rng.normal(size=128)
    B /= np.linalg.norm(np.tensordot(A, B, axes=([2], [0])))
    An, Bn, k, disc = gate(A, B, ql, qM, qr, 0, 128, 1e-13, np.cos(0.3), np.sin(0.3))
    # the gate mixes the blocks (their ranks rise above 128 in all) and keeps the norm
    assert k == 128
    assert abs(float((An ** 2).sum()) + disc - 1.0) <= 1e-12


def test_a_pair_on_a_cluster_equals_the_pair_among_many():
    """One CTA per pair (a pair list that fills the GPU) and a cluster per pair give the same bits."""
    w = inputs.make_workload(9, 4, 5, 18, 3, [24, 40, 33], seed=4)
    with tnqe.Context(w.h1, w.eri, w.N, w.n_alpha, w.n_beta) as g:
        for m in w.mps:
            g.add_mps(m.tensors, m.U)
        base = [(0, 1), (0, 2), (1, 2), (2, 0), (1, 0)]
        H1, S1 = g.matrix_elements(base)
        H2, S2 = g.matrix_elements(base * 40)
    assert np.array_equal(np.tile(H1, 40), H2) and np.array_equal(np.tile(S1, 40), S2)


@pytest.mark.parametrize("M", [1, 2, 3, 8, 31, 32])
def test_solve_sizes_match_lapack(M):
    rng = np.random.default_rng(M)
    A = rng.normal(size=(M, M))
    H = A + A.T - 20.0 * np.diag(np.arange(M))
    Y = rng.normal(size=(M, 2 * M + 2)) / np.sqrt(M)
    S = np.eye(M) + Y @ Y.T
    with tnqe.Context(np.zeros((2, 2)), np.zeros((2, 2, 2, 2)), 2, 1, 1) as g:
        E, C, r, k1 = g.solve(H, S)
    L = np.linalg.cholesky(S)
    ref = np.linalg.eigvalsh(np.linalg.solve(L, np.linalg.solve(L, H).T))
    assert r == M
    # rounding of either route: a few eps of the norms over the smallest eigenvalue of S (1)
    assert np.abs(E - ref).max() <= 64 * 2.2e-16 * M * np.abs(H).sum(0).max()
    assert np.abs(C.T @ S @ C - np.eye(M)).max() <= 64 * 2.2e-16 * M * np.abs(S).sum(0).max()
    assert np.abs(C.T @ H @ C - np.diag(E)).max() <= 64 * 2.2e-16 * M * np.abs(H).sum(0).max()


@pytest.mark.parametrize("chi", [[30, 47], [48, 71], [100, 72, 97]])
def test_contraction_items_shared_by_ctas_give_the_same_bits(chi):
    """Few pairs (up to eight CTAs per item of a contraction stage, one per 24 of the bond) and many (one)."""
    w = inputs.make_workload(8, 4, 4, 6, 3, chi, seed=7)
    with tnqe.Context(w.h1, w.eri, w.N, w.n_alpha, w.n_beta) as g:
        for m in w.mps:
            g.add_mps(m.tensors, m.U)
        base = [(i, j) for i in range(3) for j in range(3)]
        H1, S1 = g.matrix_elements(base)
        H2, S2 = g.matrix_elements(base * 30)
    assert np.array_equal(np.tile(H1, 30), H2) and np.array_equal(np.tile(S1, 30), S2)
