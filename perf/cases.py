"""What the speed of this framework is measured on: the calls that its users make, over their real range.

A case is one of five kinds of call:

* ``elements``: tnqe_matrix_elements on a list of pairs (the method's hot path:
  rotation of the kets, contraction with the Hamiltonian).  ``pairs`` is
  ``all`` (every i <= j of the M states, a whole subspace), ``row`` (one state
  against all, what a subspace that grows by one state asks for) or ``own``
  (the (i, i) pairs: energies of the states in their own orbitals, the
  contraction alone).  ``chi`` lists the bond dimensions that the states draw from.
* ``step``: one step of the generalized sweep: the states are added, R
  candidate rotations of one of them are added, their rows are computed and
  every candidate's pencil is solved (fresh states, so no captured graph).
* ``scan``: the coarse scan of the local orbital optimisation of one bond, a
  truncating two-site gate per angle, and the two-site tensor of the last angle.
* ``solve``: the generalized eigenproblem of a subspace.
* ``train``: loss and gradient of the rotation-proposal network on a batch.

Inputs are random states in the particle-number block structure that the
library requires, random symmetric integrals and random orbital rotations, with
the distributions of the framework's own workloads; the seed sets them all.
"""
import functools
import math

import numpy as np
import torch

from paper_2404_10223_gb300 import inputs, mlp, orbital_opt, sweep, tnqe

LOCAL = inputs.LOCAL_CHARGE                      # k -> (n_alpha, n_beta)


def listed():
    return [
        # the smallest subspace of the framework's workloads (N = 6, chi = 8): latency, launches, host work of a call
        dict(name="elements_n6_chi8", kind="elements", N=6, na=3, nb=3, M=3, chi="8", pairs="all", prec=0, cutoff=1e-14),
        # an ordinary small molecule (N = 10, chi = 32): 15 rotations, far fewer than there are SMs
        dict(name="elements_n10_chi32", kind="elements", N=10, na=5, nb=5, M=6, chi="32", pairs="all", prec=0, cutoff=1e-14),
        # an odd, ragged open-shell subspace: uneven spins, odd bond dimensions, an odd number of orbitals
        dict(name="elements_n11_ragged", kind="elements", N=11, na=6, nb=4, M=9, chi="13,37,61", pairs="all", prec=0, cutoff=1e-14),
        # the batched workload with uneven bond dimensions
        dict(name="elements_n14_mixed", kind="elements", N=14, na=7, nb=7, M=16, chi="32,64,128", pairs="all", prec=0, cutoff=1e-14),
        # the benchmark's workload: 136 pairs, every state at chi = 128
        dict(name="elements_n14_chi128", kind="elements", N=14, na=7, nb=7, M=16, chi="128", pairs="all", prec=0, cutoff=1e-14),
        # one state against a large-molecule subspace (N = 20, the cutoff of that workload)
        dict(name="row_n20_chi128", kind="elements", N=20, na=10, nb=10, M=9, chi="128", pairs="row", prec=0, cutoff=1e-10),
        # energies in the own orbitals on the tensor cores (sliced BF16, five slices): the contraction alone
        dict(name="own_n12_bf16x15", kind="elements", N=12, na=6, nb=6, M=8, chi="64", pairs="own", prec=5, cutoff=1e-14),
        # a step of the learned-proposal sweep: N = 12, chi = 64, 8 states, 4 candidates
        dict(name="sweep_step_n12", kind="step", N=12, na=6, nb=6, M=8, R=4, chi="64", cutoff=1e-14),
        # the scan of one bond of a chi = 64 state
        dict(name="bond_scan_chi64", kind="scan", N=12, na=6, nb=6, bond=6, chi="64", keep=64),
        # the pencil of the largest subspace of the workloads
        dict(name="solve_m24", kind="solve", M=24),
        # a training batch of the N = 12 proposal network
        dict(name="train_b512", kind="train", N=12, hidden=256, batch=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Relative cost of an elements or step case: gates times chi^2, times the waves of rotations."""
    chi = max(int(x) for x in c["chi"].split(","))
    rot = sum(i != j for i, j in _pairs(c)) if c["kind"] == "elements" else c["R"] * (c["M"] - 1)
    return c["N"] * (c["N"] - 1) / 2 * chi ** 2 * max(1.0, rot / 150.0)


def draw(rng):
    while True:
        kind = rng.choice(["elements"] * 6 + ["step", "scan", "solve", "train"])
        if kind == "solve":
            return dict(kind=kind, M=rng.randint(2, 32))
        if kind == "train":
            return dict(kind=kind, N=rng.randint(4, 16), hidden=256, batch=_log_int(rng, 16, 4096))
        N = rng.randint(5, 16)
        c = dict(kind=kind, N=N, na=min(14, max(1, N // 2 + rng.randint(-1, 1))), nb=min(14, max(1, N // 2 + rng.randint(-1, 1))),
                 chi=str(_log_int(rng, 5, 128)))
        if kind == "scan":
            return dict(c, bond=rng.randint(1, N - 1), keep=max(1, int(c["chi"]) - rng.randint(0, 3)))
        c["cutoff"] = rng.choice([1e-14, 1e-14, 1e-10])
        if kind == "step":
            c = dict(c, M=rng.randint(2, 8), R=rng.randint(1, 5))
        else:
            if rng.random() < 0.4:
                c["chi"] += "," + str(_log_int(rng, 5, 128))
            c["pairs"] = rng.choice(["all", "all", "row", "own"])
            c["M"] = rng.randint(2, 16)
            c["prec"] = rng.choice([0, 0, 5]) if c["pairs"] == "own" else 0
        if _cost(c) <= 91 * 128 ** 2:
            return c


# ----------------------------------------------------------------------------- inputs
def _pairs(c):
    M = c["M"]
    if c["pairs"] == "all":
        return [(i, j) for i in range(M) for j in range(i, M)]
    return [(M - 1, j) for j in range(M)] if c["pairs"] == "row" else [(i, i) for i in range(M)]


@functools.lru_cache(maxsize=256)
def _sectors(N, na, nb, chi):
    """Sector dimensions per bond and the charge of every index (they do not depend on the seed)."""
    secs = inputs.bond_sectors(N, na, nb, chi)
    return [{q: s[q] for q in sorted(s)} for s in secs]


def _state(rng, N, na, nb, chi):
    """A random normalised state, left-orthonormal on sites 0..N-2, indices of every bond grouped by charge."""
    secs = _sectors(N, na, nb, chi)
    offs = [dict(zip(s, np.concatenate([[0], np.cumsum(list(s.values()))[:-1]]).astype(int))) for s in secs]
    carry = {(0, 0): np.ones((1, 1))}            # R of the sites to the left, per sector
    ts = []
    for s in range(N):
        L, R = secs[s], secs[s + 1]
        T = np.zeros((sum(L.values()), 4, sum(R.values())))
        new = {}
        for q, d in R.items():
            rows = [(k, (q[0] - a, q[1] - b)) for k, (a, b) in enumerate(LOCAL) if (q[0] - a, q[1] - b) in L]
            blk = np.concatenate([carry[p] @ rng.normal(size=(L[p], d)) for _, p in rows])
            if s + 1 < N:
                blk, new[q] = np.linalg.qr(blk)
            else:
                blk = blk / np.linalg.norm(blk)
            at = 0
            for k, p in rows:
                T[offs[s][p]:offs[s][p] + L[p], k, offs[s + 1][q]:offs[s + 1][q] + d] = blk[at:at + L[p]]
                at += L[p]
        carry = new
        ts.append(T)
    return ts


def _rotation(rng, N, sigma):
    low = np.tril(rng.normal(0.0, sigma, (N, N)), -1)
    return low - low.T


def _orthogonal(K):
    return torch.linalg.matrix_exp(torch.from_numpy(K)).numpy()


def _subspace(c, seed):
    """(h1, eri, [(tensors, U)], generators) of an elements or step case."""
    rng = np.random.default_rng([seed, c["N"], c["M"]])
    h1, eri = inputs.draw_integrals(rng, c["N"], 2 * c["N"])
    chis = [int(x) for x in c["chi"].split(",")]
    states, Ks = [], []
    for j in range(c["M"]):
        K = _rotation(rng, c["N"], 0.3) if j else np.zeros((c["N"], c["N"]))
        states.append((_state(rng, c["N"], c["na"], c["nb"], chis[int(rng.integers(len(chis)))]), _orthogonal(K)))
        Ks.append(K)
    return h1, eri, states, Ks, rng


def _step_inputs(c, seed):
    h1, eri, states, Ks, rng = _subspace(c, seed)
    j = int(rng.integers(c["M"]))
    cand = [_orthogonal(Ks[j] + _rotation(rng, c["N"], 0.05)) for _ in range(c["R"])]
    M = c["M"]
    # the state that comes first in the list is the bra, as in the sweep; candidates have the ids M, M + 1, ...
    pairs = [(i, M + r) if i < j else (M + r, i) for r in range(c["R"]) for i in range(M) if i != j]
    pairs += [(M + r, M + r) for r in range(c["R"])]
    A = rng.normal(size=(M, M))
    Y = 0.01 * rng.normal(size=(M, M))
    H = np.diag(-20.0 - np.arange(M)) + 0.5 * (A + A.T)     # the subspace's stored pencil, well conditioned
    S = np.eye(M) + 0.5 * (Y + Y.T)
    return h1, eri, states, j, cand, pairs, H, S


def _scan_inputs(c, seed):
    """Two neighbouring sites with the centre on the second, random and normalised, and the bond charges."""
    rng = np.random.default_rng([seed, c["N"], c["bond"]])
    ts = _state(rng, c["N"], c["na"], c["nb"], int(c["chi"]))
    secs = _sectors(c["N"], c["na"], c["nb"], int(c["chi"]))
    A, B = ts[c["bond"] - 1], ts[c["bond"]]
    q = [[a * 16 + b for (a, b), d in secs[x].items() for _ in range(d)] for x in (c["bond"] - 1, c["bond"], c["bond"] + 1)]
    B = B * rng.uniform(0.2, 1.0, size=B.shape)              # a two-site tensor with unequal singular values
    return A, B / np.linalg.norm(B), q


def _scan_angles():
    n = orbital_opt.GRID
    return [-math.pi / 2 + k * math.pi / n for k in range(n + 1)]


def _pencil(c, seed):
    rng = np.random.default_rng([seed, c["M"]])
    M = c["M"]
    A = rng.normal(size=(M, M))
    Y = rng.normal(size=(M, M + 4)) / math.sqrt(M)
    return np.diag(-100.0 - 3.0 * np.arange(M)) + A + A.T, np.eye(M) + Y @ Y.T


def _batch(c, seed):
    rng = np.random.default_rng([seed, c["N"], c["batch"]])
    n_out = c["N"] * (c["N"] - 1) // 2
    n_in = sweep.n_features(c["N"])
    P = inputs.draw_mlp_params(rng, n_in, c["hidden"], n_out)
    X = rng.normal(0.0, 0.3, (c["batch"], n_in)).astype(np.float32)
    T = rng.normal(0.0, 0.05, (c["batch"], n_out)).astype(np.float32)
    return P, X, T, rng.exponential(0.1, c["batch"]).astype(np.float32)


# ----------------------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "elements":
        h1, eri, states, _, _ = _subspace(case, seed)
        g = tnqe.Context(h1, eri, case["N"], case["na"], case["nb"], cutoff=case["cutoff"], precision=case["prec"])
        for ts, U in states:
            g.add_mps(ts, U)
        return dict(kind=kind, g=g, pairs=_pairs(case))
    if kind == "step":
        h1, eri, states, j, cand, pairs, H, S = _step_inputs(case, seed)
        b = sweep.LibraryBackend(h1, eri, case["N"], case["na"], case["nb"], cutoff=case["cutoff"], use_graphs=0)
        return dict(kind=kind, b=b, states=states, j=j, cand=cand, pairs=pairs, H=H, S=S)
    if kind == "scan":
        A, B, q = _scan_inputs(case, seed)
        return dict(kind=kind, o=orbital_opt.BondOptimizer(A, B, *q, case["keep"]), shape=(A.shape[0], B.shape[2]))
    if kind == "solve":
        H, S = _pencil(case, seed)
        return dict(kind=kind, H=H, S=S, g=tnqe.Context(np.zeros((2, 2)), np.zeros((2, 2, 2, 2)), 2, 1, 1))
    P, X, T, w = _batch(case, seed)
    net = mlp.Mlp(X.shape[1], case["hidden"], T.shape[1], max_batch=case["batch"])
    net.set_params(P)
    return dict(kind=kind, net=net, X=X, T=T, w=w)


def run(state):
    kind = state["kind"]
    if kind == "elements":
        return state["g"].matrix_elements(state["pairs"])
    if kind == "step":
        b, M, j = state["b"], len(state["states"]), state["j"]
        b.reset()
        for ts, U in state["states"]:
            b.add_mps(ts, U)
        for U in state["cand"]:
            b.add_mps(state["states"][j][0], U)
        Hv, Sv = b.matrix_elements(state["pairs"])
        others = [i for i in range(M) if i != j]
        E = []
        for r in range(len(state["cand"])):
            H, S = state["H"].copy(), state["S"].copy()
            H[others, j] = H[j, others] = Hv[r * (M - 1):(r + 1) * (M - 1)]
            S[others, j] = S[j, others] = Sv[r * (M - 1):(r + 1) * (M - 1)]
            H[j, j], S[j, j] = Hv[len(state["cand"]) * (M - 1) + r], Sv[len(state["cand"]) * (M - 1) + r]
            E.append(b.energies(H, S))
        return Hv, Sv, np.array(E)
    if kind == "scan":
        xi = []
        for t in _scan_angles():
            x, An, Bn, q = state["o"].apply(t)
            xi.append(x)
        return np.array(xi), np.asarray(q), np.tensordot(An, Bn, axes=([2], [0]))
    if kind == "solve":
        return state["g"].solve(state["H"], state["S"])
    return state["net"].gradient(state["X"], state["T"], state["w"])


# ----------------------------------------------------------------------------- what a pass cannot do without
def _channels(N, b):
    """(charge change, number of MPO channels) of bond b: the identity and the completed Hamiltonian, one- and three-operator
    strings, and the operator pairs of the shorter side."""
    h = min(b, N - b)
    out = {(0, 0): 2.0 + 2 * h * h}
    for d, n in [((1, 0), N), ((-1, 0), N), ((0, 1), N), ((0, -1), N), ((1, -1), h * h), ((-1, 1), h * h), ((1, 1), h * h),
                 ((-1, -1), h * h)] + [((2 * x, 0), h * (h - 1) / 2) for x in (1, -1)] + [((0, 2 * x), h * (h - 1) / 2) for x in (1, -1)]:
        out[d] = out.get(d, 0.0) + n
    return out


@functools.lru_cache(maxsize=256)
def _pair_flops(N, na, nb, chi_i, chi_j, rotated):
    """FLOPs of one pair in charge blocks of the input sector dimensions: the two environment products of every site and,
    for a rotated pair, each gate's two-site product, gate and block SVDs (4 m n^2 + 8 n^3 per m x n block)."""
    A, B = _sectors(N, na, nb, chi_i), _sectors(N, na, nb, chi_j)
    fl = 0.0
    for t in range(N):
        for (d, Dc) in _channels(N, t).items():
            for q, a in A[t].items():
                p = (q[0] - d[0], q[1] - d[1])
                if p in B[t]:
                    fl += 2.0 * a * Dc * B[t][p] * sum(B[t + 1].get((p[0] + x, p[1] + y), 0) for x, y in LOCAL)
        for (d, Dc) in _channels(N, t + 1).items():
            for q, a in A[t + 1].items():
                p = (q[0] - d[0], q[1] - d[1])
                fl += 2.0 * a * Dc * B[t + 1].get(p, 0) * sum(A[t].get((q[0] - x, q[1] - y), 0) for x, y in LOCAL)
    if rotated:
        per = [0.0] * (N - 1)
        for s in range(N - 1):
            per[s] = _gate_flops(B[s], B[s + 1], B[s + 2])
        # the plan's gate p is applied min(p, N - 2 - p) + ... times: every sweep k acts on the sites that are left
        lo, hi, top = 0, N - 1, True
        while lo < hi:
            fl += sum(per[lo:hi])
            lo, hi, top = (lo + 1, hi, False) if top else (lo, hi - 1, True)
    return fl


def _gate_flops(L, Mid, R):
    fl = 0.0
    for q, l in L.items():
        for x, y in LOCAL:
            m = Mid.get((q[0] + x, q[1] + y), 0)
            fl += sum(2.0 * l * m * R.get((q[0] + x + u, q[1] + y + v), 0) for u, v in LOCAL)
    for q in {(q[0] + x, q[1] + y) for q in L for x, y in LOCAL}:
        r = sum(L.get((q[0] - x, q[1] - y), 0) for x, y in LOCAL)
        c = sum(R.get((q[0] + x, q[1] + y), 0) for x, y in LOCAL)
        m, n = max(r, c), min(r, c)
        fl += 4.0 * m * n * n + 8.0 * n ** 3 + 8.0 * m * n
    return fl


def _state_bytes(N, na, nb, chi):
    s = _sectors(N, na, nb, chi)
    return sum(8.0 * l * sum(s[t + 1].get((q[0] + x, q[1] + y), 0) for x, y in LOCAL) for t in range(N) for q, l in s[t].items())


def work(case):
    kind = case["kind"]
    if kind == "solve":
        M = case["M"]
        return {"bytes": 8.0 * (3 * M * M + M), "flops": 2 * 9.0 * M ** 3 + 6.0 * M ** 3}
    if kind == "train":
        n_in, n_out, h, B = sweep.n_features(case["N"]), case["N"] * (case["N"] - 1) // 2, case["hidden"], case["batch"]
        mac = n_in * h + h * h + h * n_out
        return {"bytes": 4.0 * (B * (n_in + n_out + 1) + 2 * mac), "flops": 2.0 * B * (3 * mac - n_in * h)}
    if kind == "scan":
        s = _sectors(case["N"], case["na"], case["nb"], int(case["chi"]))
        L, Mid, R = s[case["bond"] - 1], s[case["bond"]], s[case["bond"] + 1]
        dims = [sum(x.values()) for x in (L, Mid, R)]
        n = len(_scan_angles())
        return {"bytes": 8.0 * 4 * dims[1] * (dims[0] + dims[2]) * (1 + n), "flops": n * _gate_flops(L, Mid, R)}
    N, na, nb = case["N"], case["na"], case["nb"]
    chis = [int(x) for x in case["chi"].split(",")]

    def mean(f):                                   # over the bond dimensions that the states draw from
        return sum(f(a, b) for a in chis for b in chis) / len(chis) ** 2

    if kind == "step":
        rot, own, M = case["R"] * (case["M"] - 1), case["R"], case["M"] + case["R"]
    else:
        pl = _pairs(case)
        rot, M = sum(i != j for i, j in pl), case["M"]
        own = len(pl) - rot
    fl = rot * mean(lambda a, b: _pair_flops(N, na, nb, a, b, True)) + own * mean(lambda a, b: _pair_flops(N, na, nb, a, a, False))
    return {"bytes": M * mean(lambda a, b: _state_bytes(N, na, nb, a)) + 16.0 * (rot + own), "flops": fl}


# ----------------------------------------------------------------------------- the same in 64 bits
def _givens(V):
    """Nearest-neighbour rotations (site, c, s, side) of V in the order of application, and the site of a sign or -1."""
    W, N = np.array(V), V.shape[0]
    lo, hi, top, passes = 0, N - 1, True, []
    while lo < hi:
        this = []
        for a in (range(hi - 1, lo - 1, -1) if top else range(lo, hi)):
            x, y = W[lo if top else hi, a], W[lo if top else hi, a + 1]
            r = math.hypot(x, y)
            c, s = (1.0, 0.0) if r < 1e-14 else (x / r, y / r) if top else (y / r, -x / r)
            W[:, [a, a + 1]] = W[:, [a, a + 1]] @ np.array([[c, -s], [s, c]])
            this.append([a, c, s, 0 if top else 1])
        lo, hi, top = (lo + 1, hi, False) if top else (lo, hi - 1, True)
        passes.append(this)
    for this in passes[:-1]:
        this[-1][3] ^= 1                          # the centre turns toward the next pass
    return [g for this in passes for g in this], (lo if W[lo, lo] < 0 else -1)


def _gate(c, s):
    """exp(theta sum_s (a+_0s a_1s - a+_1s a_0s)) on the modes 0a 0b 1a 1b, index 4 k0 + k1."""
    ops = []
    for j in range(4):
        m = np.zeros((16, 16))
        for K in range(16):
            n = [K >> 2 & 1, K >> 3 & 1, K & 1, K >> 1 & 1]
            if n[j]:
                n2 = [x if i != j else 0 for i, x in enumerate(n)]
                m[4 * (n2[0] + 2 * n2[1]) + n2[2] + 2 * n2[3], K] = (-1) ** sum(n[:j])
        ops.append(m)
    T = sum(ops[i].T @ ops[2 + i] - ops[2 + i].T @ ops[i] for i in (0, 1))
    return torch.linalg.matrix_exp(torch.from_numpy(math.atan2(s, c) * T)).numpy()


def _split(theta, keep, cutoff):
    """Truncated SVD of a two-site tensor: (u, sigma, vt, discarded weight)."""
    m = theta.reshape(theta.shape[0] * 4, -1)
    u, sg, vt = np.linalg.svd(m, full_matrices=False)
    k = max(1, min(keep, int((sg > cutoff * sg[0]).sum())))
    return u[:, :k].reshape(theta.shape[0], 4, k), sg[:k], vt[:k].reshape(k, 4, -1), float((sg[k:] ** 2).sum())


def _rotated(ts, V, keep, cutoff):
    ts = list(ts)
    gates, neg = _givens(V)
    for a, c, s, side in gates:
        th = np.einsum("xyab,labr->lxyr", _gate(c, s).reshape(4, 4, 4, 4), np.tensordot(ts[a], ts[a + 1], axes=([2], [0])))
        u, sg, vt, _ = _split(th, keep, cutoff)
        ts[a], ts[a + 1] = (u * sg, vt) if side == 0 else (u, sg[:, None, None] * vt)
    if neg >= 0:
        ts[neg] = ts[neg] * np.array([1.0, -1.0, -1.0, 1.0])[None, :, None]
    return ts


@functools.lru_cache(maxsize=8)
def _strings(N, n):
    """Occupation strings of n particles, and for every (p, q): source string and sign of a+_p a_q."""
    st = [x for x in range(1 << N) if bin(x).count("1") == n]
    at = {x: i for i, x in enumerate(st)}
    src, sgn = np.zeros((N, N, len(st)), dtype=np.int64), np.zeros((N, N, len(st)))
    for i, x in enumerate(st):
        for p in range(N):
            for q in range(N):                    # result string x = a+_p a_q y
                if x >> p & 1 and (p == q or not x >> q & 1):
                    y = x ^ (1 << p) ^ (1 << q) if p != q else x
                    lo, hi = min(p, q), max(p, q)
                    src[p, q, i] = at[y]
                    sgn[p, q, i] = (-1) ** bin(x >> (lo + 1) & ((1 << max(0, hi - lo - 1)) - 1)).count("1")
    return st, src, sgn


def _vector(ts, N, na, nb):
    """The state as a (alpha string, beta string) matrix, all alpha creators first."""
    v = np.ones((1, 1))
    half = N // 2
    parts = []
    for a, b in ((0, half), (half, N)):
        v = ts[a]
        v = v.reshape(v.shape[0], -1, v.shape[2])
        for t in ts[a + 1:b]:
            v = np.tensordot(v, t, axes=([2], [0])).reshape(v.shape[0], -1, t.shape[2])
        parts.append(v)
    sa, sb = _strings(N, na)[0], _strings(N, nb)[0]
    kidx = np.array([[[(x >> p & 1) + 2 * (y >> p & 1) for p in range(N)] for y in sb] for x in sa])
    left = kidx[:, :, :half] @ (4 ** np.arange(half - 1, -1, -1))
    right = kidx[:, :, half:] @ (4 ** np.arange(N - half - 1, -1, -1))
    full = torch.from_numpy(parts[0][0]).cuda() @ torch.from_numpy(parts[1][:, :, 0]).cuda()
    sign = np.array([[(-1) ** sum(bin(y & ((1 << p) - 1)).count("1") for p in range(N) if x >> p & 1) for y in sb] for x in sa])
    return full[torch.from_numpy(left).cuda(), torch.from_numpy(right).cuda()] * torch.from_numpy(sign).double().cuda()


def _excite(C, N, na, nb):
    """E_pq C for every (p, q): (N^2, strings, strings)."""
    _, ia, ga = _strings(N, na)
    _, ib, gb = _strings(N, nb)
    n = N * N
    ia, ga, ib, gb = (torch.from_numpy(x.reshape(n, -1)).cuda() for x in (ia, ga, ib, gb))
    return C[ia] * ga[:, :, None] + (C[:, ib] * gb[None]).permute(1, 0, 2)


def _exact_pairs(c, h1, eri, states, pairs):
    N, na, nb, cutoff = c["N"], c["na"], c["nb"], c["cutoff"]
    H, S = [], []
    bras, kets = {}, {}
    for i, j in pairs:
        ti, Ui = states[i]
        tj, Uj = states[j]
        if i not in bras:
            h = Ui.T @ h1 @ Ui
            g = eri
            for _ in range(4):
                g = np.tensordot(g, Ui, axes=([0], [0]))
            b = _vector(ti, N, na, nb)
            eb = _excite(b, N, na, nb).reshape(N, N, -1).transpose(0, 1).reshape(N * N, -1)   # E_qp bra at (p, q)
            one = h - 0.5 * np.einsum("pqqs->ps", g)
            bras[i] = (b, eb, torch.from_numpy(one.ravel()).cuda(), torch.from_numpy(0.5 * g.reshape(N * N, N * N)).cuda())
        b, eb, one, two = bras[i]
        k = _vector(tj if i == j else _rotated(tj, Ui.T @ Uj, max(t.shape[2] for t in tj), cutoff), N, na, nb)
        ek = _excite(k, N, na, nb).reshape(N * N, -1)
        H.append(float(one @ (ek @ b.reshape(-1)) + (two * (eb @ ek.T)).sum()))
        S.append(float((b * k).sum()))
    return np.array(H), np.array(S)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        H, S = _pencil(case, seed)
        lam, W = np.linalg.eigh(S)
        X = W / np.sqrt(lam)
        E, Y = np.linalg.eigh(X.T @ H @ X)
        C = X @ Y
        C = C * np.where(np.take_along_axis(C, np.abs(C).argmax(0)[None], 0) < 0, -1.0, 1.0)
        return E, C, case["M"], float(C[:, 0] @ C[:, 0] / math.sqrt(E[0] ** 2 + 1.0))
    if kind == "train":
        P, X, T, w = (torch.from_numpy(x).double() for x in _batch(case, seed))
        n_in, n_out, h = X.shape[1], T.shape[1], case["hidden"]
        P.requires_grad_(True)
        W1, b1, W2, b2, W3, b3 = torch.split(P, [h * n_in, h, h * h, h, n_out * h, n_out])
        f = torch.nn.functional
        Y = f.linear(f.gelu(f.linear(f.gelu(f.linear(X, W1.view(h, n_in), b1)), W2.view(h, h), b2)), W3.view(n_out, h), b3)
        loss = (w[:, None] * (Y - T) ** 2).sum() / (w.sum() * n_out)
        loss.backward()
        return float(loss.detach()), P.grad.numpy()
    if kind == "scan":
        A, B, _ = _scan_inputs(case, seed)
        xi = []
        for t in _scan_angles():
            th = np.einsum("xyab,labr->lxyr", _gate(math.cos(t), math.sin(t)).reshape(4, 4, 4, 4), np.tensordot(A, B, axes=([2], [0])))
            u, sg, vt, disc = _split(th, case["keep"], 0.0)
            xi.append(disc / (disc + float((sg ** 2).sum())))
        return np.array(xi), None, np.tensordot(u * sg, vt, axes=([2], [0]))
    # the elements of a subspace by its vectors in the Fock sector: as long as these, and the dense SVDs, are small
    chi = max(int(x) for x in case["chi"].split(","))
    strings = math.comb(case["N"], case["na"]) * math.comb(case["N"], case["nb"])
    if kind == "step" or strings > 1e6 or case["M"] > 9:
        return None
    pairs = _pairs(case)
    rot = sum(i != j for i, j in pairs)
    if rot * case["N"] ** 2 / 2 * (4.0 * chi) ** 3 * 2e-9 > 15 or (case["M"] + len(pairs)) * strings > 2.5e7:
        return None
    h1, eri, states, _, _ = _subspace(case, seed)
    return _exact_pairs(case, h1, eri, states, pairs)
