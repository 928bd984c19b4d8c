"""The gate's truncation at the ends of its arguments' ranges (tnqe_apply_gate_noalloc with the identity gate on blocks
of chosen size and spectrum), against NumPy's SVD or against the same call in the middle of the range."""
import numpy as np
import pytest

from paper_2404_10223_gb300 import inputs, tnqe

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import os
    from paper_2404_10223_gb300 import build as B
    if not os.path.exists(B.LIB):
        B.build()
    tnqe.load()


def gate(A, B, q, side, chi_max, cutoff):
    import torch
    dA, dB = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B))
    chl, chm, chr_ = A.shape[0], A.shape[2], B.shape[2]
    Ao = torch.zeros(chl * 4 * chi_max, dtype=torch.float64, device="cuda")
    Bo = torch.zeros(chi_max * 4 * chr_, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    k, _, disc = tnqe.tnqe_apply_gate_noalloc(dA.data_ptr(), dB.data_ptr(), chl, chm, chr_, *q, 1.0, 0.0, side,
                                              chi_max, cutoff, 60, Ao.data_ptr(), Bo.data_ptr(), 0)
    return (Ao[: chl * 4 * k].cpu().numpy().reshape(chl, 4, k), Bo[: k * 4 * chr_].cpu().numpy().reshape(k, 4, chr_),
            k, disc)


def blocks(shapes, spectra, rng):
    """A two-site tensor with one block per (rows, cols), local states 3, 3, charges that do not couple."""
    rows, cols, rs = ([0] + list(np.cumsum(x)) for x in
                      ([s[0] for s in shapes], [s[1] for s in shapes], [len(x) for x in spectra]))
    A, B = np.zeros((rows[-1], 4, rs[-1])), np.zeros((rs[-1], 4, cols[-1]))
    q = [[], [], []]
    for b, ((m, n), sg) in enumerate(zip(shapes, spectra)):
        r = len(sg)
        A[rows[b]:rows[b + 1], 3, rs[b]:rs[b + 1]] = np.linalg.qr(rng.normal(size=(m, r)))[0]
        B[rs[b]:rs[b + 1], 3, cols[b]:cols[b + 1]] = np.asarray(sg)[:, None] * np.linalg.qr(rng.normal(size=(n, r)))[0].T
        for x, (base, count) in enumerate([(17, m), (34, r), (51, n)]):
            q[x] += [base + 3 * b] * count
    return A, B, q


@pytest.mark.parametrize("cutoff", [1.0, 1.5, 10.0, 1e300])
@pytest.mark.parametrize("n", [4, 24, 90])
@pytest.mark.parametrize("side", [0, 1])
def test_a_cutoff_of_one_and_more_keeps_the_largest_singular_value(cutoff, n, side):
    rng = np.random.default_rng(n)
    A, B, q = blocks([(n + 3, n)], [1.0 - 0.9 * np.arange(n) / n], rng)
    An, Bn, k, disc = gate(A, B, q, side, n, cutoff)
    th = np.tensordot(A, B, axes=([2], [0]))[:, 3, 3, :]
    u, sg, vt = np.linalg.svd(th)
    assert k == 1
    # FP64 rounding of either SVD over the gap at the cut (0.9 / n)
    assert np.abs(np.tensordot(An, Bn, axes=([2], [0]))[:, 3, 3, :] - sg[0] * np.outer(u[:, 0], vt[0])).max() <= 1e-15 * n ** 2
    assert abs(disc - (sg[1:] ** 2).sum()) <= 1e-12 * n


@pytest.mark.parametrize("cutoff", [0.5, 1.0, 2.0])
def test_a_cutoff_of_one_and_more_compares_narrow_and_wide_blocks(cutoff):
    rng = np.random.default_rng(3)
    A, B, q = blocks([(5, 4), (30, 24), (6, 4)], [[0.9, 0.3, 0.2, 0.1], np.linspace(1.0, 0.1, 24), [0.8, 0.1, 0.1, 0.05]], rng)
    An, Bn, k, _ = gate(A, B, q, 0, 64, cutoff)
    s = np.concatenate([[0.9, 0.3, 0.2, 0.1], np.linspace(1.0, 0.1, 24), [0.8, 0.1, 0.1, 0.05]])
    kept = np.sort(np.linalg.norm(An.reshape(-1, k), axis=0))[::-1]
    ref = np.sort(s)[::-1][: max(1, int((s > cutoff).sum()))]
    assert k == len(ref) and np.abs(kept - ref).max() <= 1e-14


@pytest.mark.parametrize("cutoff", [float("nan"), 1.5, 1e200])
def test_rotations_with_such_a_cutoff_keep_one_column_a_bond(cutoff):
    w = inputs.make_workload(6, 3, 3, 12, 2, [16, 16], seed=5)
    ref = None
    for ct in (1.0 - 1e-9, cutoff):                  # below 1 by less than any gap: the largest alone is above it
        with tnqe.Context(w.h1, w.eri, w.N, w.n_alpha, w.n_beta, cutoff=ct) as g:
            for m in w.mps:
                g.add_mps(m.tensors, m.U)
            g.rotate(0, 1)
            got = g.get_rotated()
        assert all(t.shape[2] == 1 for t in got)
        if ref is not None:
            assert all(np.array_equal(a, b) for a, b in zip(ref, got))
        ref = got


@pytest.mark.parametrize("e", [-900, -600, -450, 450, 600, 900, 1000])
@pytest.mark.parametrize("n", [4, 24, 60, 90])
@pytest.mark.parametrize("side", [0, 1])
def test_a_tensor_times_a_power_of_two_gives_the_same_bits(e, n, side):
    """The squares of the singular values leave the range of FP64 beyond 2^+-512; the singular values do not."""
    rng = np.random.default_rng(n)
    two = 2 if n <= 60 else 1                         # bonds of up to 128
    A, B, q = blocks([(n + 3, n), (n, n + 2)][:two], [1.0 - 0.9 * np.arange(n) / n, 0.7 - 0.6 * np.arange(n) / n][:two], rng)
    keep = n // 2 + 1
    An, Bn, k, disc = gate(A, B, q, side, keep, 1e-14)
    As, Bs, ks, ds = gate(np.ldexp(A, e), B, q, side, keep, 1e-14)
    assert k == ks == keep
    # the factor with the singular values takes the power of two
    assert np.array_equal(np.ldexp(An, e if side == 0 else 0), As) and np.array_equal(np.ldexp(Bn, e if side == 1 else 0), Bs)
    if abs(e) < 500:
        assert ds == np.ldexp(disc, 2 * e)


@pytest.mark.parametrize("n", [2, 4, 5, 8, 9, 24, 60, 90])
@pytest.mark.parametrize("close", [1e-3, 1e-6, 1e-9])
@pytest.mark.parametrize("tall", [False, True])
@pytest.mark.parametrize("side", [0, 1])
def test_pairs_of_close_singular_values_leave_both_factors_orthogonal(n, close, tall, side):
    """The isometric factor is V of the block for one orientation and W / sigma for the other."""
    worst = 0.0
    for seed in range(12 if n < 10 else 3):
        rng = np.random.default_rng([n, seed])
        sg = np.linspace(1.0, 0.2, n)
        sg[1::2] = sg[0:2 * (n // 2):2] * (1.0 - close)
        A, B, q = blocks([(n + 3, n) if tall else (n, n + 3)], [sg], rng)
        An, Bn, k, _ = gate(A, B, q, side, n, 1e-14)
        assert k == n
        th = np.tensordot(A, B, axes=([2], [0]))
        assert np.abs(np.tensordot(An, Bn, axes=([2], [0])) - th).max() <= 1e-15 * (n + 3)
        X = Bn.reshape(k, -1) if side == 0 else An.reshape(-1, k).T
        worst = max(worst, np.abs(X @ X.T - np.eye(k)).max())
    # pairs are rotated down to m eps, and the last sweep leaves as much; W of wider blocks is a double-float product
    assert worst <= 4.0 * (n + 3) * 2.0 ** -52 + (n > 8) * 4.0 * 2.0 ** -48


@pytest.mark.parametrize("n", [9, 12, 24, 40, 60, 90])
@pytest.mark.parametrize("tall", [False, True])
@pytest.mark.parametrize("side", [0, 1])
def test_truncated_factors_are_orthonormal_to_fp64(n, tall, side):
    """Well separated singular values, a third of them kept: what is rounded is FP64 vectors of unit length (an error of
    2^-53 of each entry, sums of n terms in random order)."""
    rng = np.random.default_rng(n)
    sg = 1.0 - 0.9 * np.arange(n) / n
    A, B, q = blocks([(n + 3, n) if tall else (n, n + 3)], [sg], rng)
    An, Bn, k, disc = gate(A, B, q, side, n // 3, 1e-14)
    X = (Bn.reshape(k, -1) if side == 0 else An.reshape(-1, k).T).astype(np.longdouble)
    W = (An.reshape(-1, k).T if side == 0 else Bn.reshape(k, -1)).astype(np.longdouble)
    assert np.abs(X @ X.T - np.eye(k)).max() <= 2.0 ** -52 * np.sqrt(n)
    G = W @ W.T
    d = np.sqrt(np.diag(G))
    assert np.abs(d - sg[:k]).max() <= 2.0 ** -52 * np.sqrt(n)     # the tensor itself is rounded as much
    # the inner products of W are those of X times the squares of the singular values (at most 1, at least 0.46)
    assert np.abs(G / np.outer(d, d) - np.eye(k)).max() <= 2.0 ** -51 * np.sqrt(n)


def dropped_weight(m, X):
    """|m - m P|^2 in extended precision, P the projector on the rows of X: an error of X enters squared."""
    m, X = m.astype(np.longdouble), X.astype(np.longdouble)
    for _ in range(2):
        X = 1.5 * X - 0.5 * (X @ X.T) @ X
    return float(((m - (m @ X.T) @ X) ** 2).sum())


@pytest.mark.parametrize("n", [5, 9, 24, 40, 60, 90])
@pytest.mark.parametrize("low", [0.3, 0.03, 0.011])
@pytest.mark.parametrize("side", [0, 1])
def test_a_small_discarded_weight_is_as_accurate_as_a_large_one(n, low, side):
    """Kept singular values from 1 to 0.5, dropped ones around `low`: down to 2e-4 of the weight is dropped."""
    rng = np.random.default_rng([n, side])
    k = max(1, n // 3)
    sg = np.concatenate([np.linspace(1.0, 0.5, k), low * np.linspace(1.0, 0.5, n - k)])
    # the isometric factor holds the kept vectors: B for side 0, A for side 1
    A, B, q = blocks([(n + 3, n) if side == 0 else (n, n + 3)], [sg], rng)
    An, Bn, kn, disc = gate(A, B, q, side, k, 1e-14)
    th = np.tensordot(A, B, axes=([2], [0]))
    assert kn == k
    if side == 0:
        ref = dropped_weight(th.reshape(th.shape[0] * 4, -1), Bn.reshape(k, -1))
    else:
        ref = dropped_weight(th.reshape(th.shape[0] * 4, -1).T, An.reshape(-1, k).T)
    # FP64 entries of the remainder, off by 2^-53 of the block's norm (at most sqrt(k)) each, against its norm
    assert abs(disc - ref) <= 4.0 * 2.0 ** -53 * np.sqrt(k / ref) * ref


def test_a_block_that_is_discarded_whole_counts_with_its_norm():
    rng = np.random.default_rng(1)
    for n in (5, 24, 40):
        A, B, q = blocks([(60, 50), (n + 2, n)], [np.linspace(1.0, 0.5, 50), 1e-3 * np.linspace(1.0, 0.5, n)], rng)
        _, _, k, disc = gate(A, B, q, 0, 50, 1e-14)
        th = np.tensordot(A[60:], B[:, :, 50:], axes=([2], [0])).astype(np.longdouble)
        ref = float((th ** 2).sum())
        # the first block keeps all of its columns
        assert k == 50 and abs(disc - ref) <= 8.0 * 2.0 ** -53 * ref


def test_blocks_for_eight_warps_give_the_same_bits_on_every_team():
    """Blocks of 75 to 104 columns: a pair on a cluster, on one CTA among many, and run again."""
    w = inputs.make_workload(8, 4, 4, 6, 3, [150, 190, 170], seed=11)
    with tnqe.Context(w.h1, w.eri, w.N, w.n_alpha, w.n_beta) as g:
        for m in w.mps:
            g.add_mps(m.tensors, m.U)
        base = [(0, 1), (0, 2), (1, 2), (2, 0), (1, 0)]
        H1, S1 = g.matrix_elements(base)
        H2, S2 = g.matrix_elements(base * 40)
        weights = [[g.rotate(i, j) for i, j in base] for _ in range(3)]
    assert np.array_equal(np.tile(H1, 40), H2) and np.array_equal(np.tile(S1, 40), S2)
    assert weights[0] == weights[1] == weights[2]


@pytest.mark.parametrize("shapes", [[(100, 100)], [(90, 80), (30, 44)], [(52, 52), (60, 74)], [(64, 49), (50, 50)]])
@pytest.mark.parametrize("keep", [1.0, 0.7])
def test_wide_blocks_of_which_most_is_kept(shapes, keep):
    rng = np.random.default_rng(2)
    A, B, q = blocks(shapes, [np.linspace(1.0 - 0.05 * i, 0.3, min(s)) for i, s in enumerate(shapes)], rng)
    k = int(keep * sum(min(s) for s in shapes))
    th = np.tensordot(A, B, axes=([2], [0]))[:, 3, 3, :]
    sg = np.linalg.svd(th, compute_uv=False)
    first = None
    for _ in range(3):
        An, Bn, kn, disc = gate(A, B, q, 0, k, 1e-14)
        assert kn == k
        if first is None:
            first = An, Bn, disc
            X = Bn.reshape(k, -1)
            assert np.abs(X @ X.T - np.eye(k)).max() <= 2.0 ** -51 * np.sqrt(128)
            assert np.abs(np.sort(np.linalg.norm(An.reshape(-1, k), axis=0))[::-1] - sg[:k]).max() <= 2.0 ** -50 * np.sqrt(128)
        assert np.array_equal(first[0], An) and np.array_equal(first[1], Bn) and first[2] == disc


@pytest.mark.parametrize("n", [1, 2, 8, 9, 24, 60, 90, 120])
@pytest.mark.parametrize("coupling", [0.0, 1e-13, 1e-8, 1e-5])
@pytest.mark.parametrize("side", [0, 1])
def test_columns_that_are_nearly_orthogonal_already(n, coupling, side):
    """Columns of lengths 0.2 to 1 in mixed order whose inner products are about `coupling`."""
    rng = np.random.default_rng([n, side])
    d = rng.permutation(np.linspace(1.0, 0.2, n))
    M = np.linalg.qr(rng.normal(size=(n + 3, n)))[0] * d
    M = M @ (np.eye(n) + coupling * rng.normal(size=(n, n)))
    A, B = np.zeros((n + 3, 4, n)), np.zeros((n, 4, n))
    A[:, 3], B[:, 3] = M, np.eye(n)
    keep = max(1, n // 2)
    An, Bn, k, disc = gate(A, B, ([17] * (n + 3), [34] * n, [51] * n), side, keep, 1e-14)
    u, sg, vt = np.linalg.svd(M, full_matrices=False)
    assert k == keep
    X = Bn.reshape(k, -1) if side == 0 else An.reshape(-1, k).T
    # the Jacobi SVD: pairs rotated down to m eps
    assert np.abs(X @ X.T - np.eye(k)).max() <= 4.0 * (n + 3) * 2.0 ** -52
    new = np.tensordot(An, Bn, axes=([2], [0]))[:, 3, 3, :]
    gap = 0.8 / max(1, n - 1) if keep < n else 1.0
    assert np.abs(new - (u[:, :k] * sg[:k]) @ vt[:k]).max() <= 4.0 * (n + 3) * 2.0 ** -52 / gap
    assert abs(disc - (sg[k:] ** 2).sum()) <= 64 * 2.0 ** -53 * n


@pytest.mark.parametrize("zero", [(), (0,), (1,), (0, 2), (0, 1, 2)])
@pytest.mark.parametrize("shapes", [[(1, 1), (1, 1), (1, 1)], [(8, 8), (3, 2), (5, 7)], [(40, 8), (1, 8), (2, 30)],
                                    [(12, 9), (3, 3), (1, 1)]])
@pytest.mark.parametrize("side", [0, 1])
def test_gates_of_narrow_blocks_alone_some_of_them_zero(zero, shapes, side):
    """Blocks of up to 8 columns are done in the first phase (the last set has one of 9); zero blocks have no values."""
    rng = np.random.default_rng(4)
    gate(*blocks([(20, 20), (9, 9)], [np.linspace(1.0, 0.1, 20), np.linspace(1.0, 0.1, 9)], rng), side, 9, 0.0)   # other values in the scratch
    spectra = [np.zeros(min(s)) if b in zero else 1.0 - 0.07 * b - 0.8 * np.arange(min(s)) / min(s) for b, s in enumerate(shapes)]
    A, B, q = blocks(shapes, spectra, rng)
    values = np.sort(np.concatenate(spectra))[::-1]
    keep = max(2, len(values) // 2)
    An, Bn, k, disc = gate(A, B, q, side, keep, 1e-14)
    assert k == min(keep, max(1, int((values > 0).sum())))
    th = np.tensordot(A, B, axes=([2], [0]))[:, 3, 3, :]
    u, sg, vt = np.linalg.svd(th)
    got = np.tensordot(An, Bn, axes=([2], [0]))[:, 3, 3, :]
    # FP64 rounding of sums over up to 40 entries, over gaps of 0.01 and more at the cut
    assert np.abs(got - (u[:, :k] * sg[:k]) @ vt[:k]).max() <= 2e-13
    assert abs(disc - (values[k:] ** 2).sum()) <= 1e-14 * len(values)
