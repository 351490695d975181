"""Workloads of the SP-MPS library as its users call it, with plain 64-bit references.

Four kinds of call carry the framework:

* ``action``: one projected action y = H_eff x, z = N_eff x at a pair of sites (what a Davidson
  iteration, or a caller with an eigensolver of its own, issues thousands of times);
* ``step``: a state from host memory and one two-site optimisation step on it;
* ``sweep``: a state from host memory and one full two-site sweep;
* ``load``: a raw state from host memory, canonicalised on the GPU, and its energy, <P> and <S^2>.

Sizes are those of the tests (L = 6 .. 8, D = 12 .. 64), of the benchmark (L = 24, D = 256,
n_beta = 8, S = 0 and S = 1) and of the K = 20, N = 30, n_beta = 12 active-space workload.  States are
seeded random (N, M)-symmetric MPS, isometric on both sides of the pair of an action or a step.  Their
bond dimension is spread over the labels (n, 2m) as in a random initial state (in proportion to the Fock
sectors) or, ``settled``, as in an optimised one: few labels around the mean particle number, with the
larger blocks that sweeps end up with (the benchmark's middle pair has 58 to 73 thousand entries).
"""
import math

import numpy as np
import torch

_N = (0, 1, 1, 2)    # particle number and twice Sz of the local states {0, b, a, ab}
_M = (0, -1, 1, 0)


def listed():
    hub = {"kind": "action", "ham": "hubbard", "U": 4.0, "tc": False, "out": "yz"}
    return [
        # one action of the smallest workload of the tests: launches and latency count
        {**hub, "name": "action_L8_D32", "K": 8, "N": 8, "twoM": 0, "twoS": 0, "D": 32, "n_beta": 5, "site": 3},
        # odd electron number, quartet target, ragged blocks, off the middle
        {**hub, "name": "action_L13_D77_odd", "K": 13, "N": 11, "twoM": 1, "twoS": 3, "D": 77, "n_beta": 5,
         "site": 4, "U": 2.5},
        # the benchmark's action with the default options (FP64 pipe)
        {**hub, "name": "action_L24_D256", "K": 24, "N": 24, "twoM": 0, "twoS": 0, "D": 256, "n_beta": 8, "site": 11, "settled": True},
        # the same for the triplet target with the products on the tensor cores
        {**hub, "name": "action_L24_D256_S1_tc", "K": 24, "N": 24, "twoM": 2, "twoS": 2, "D": 256, "n_beta": 8,
         "site": 11, "tc": True, "settled": True},
        # metric product alone (the CG correction issues these), off the middle, tensor cores
        {**hub, "name": "metric_L24_D200_tc", "K": 24, "N": 24, "twoM": 0, "twoS": 0, "D": 200, "n_beta": 8,
         "site": 8, "tc": True, "out": "z", "settled": True},
        # active-space integrals, K = 20: the largest operator
        {**hub, "name": "action_K20_D100_ab_initio", "ham": "ab_initio", "K": 20, "N": 30, "twoM": 10, "twoS": 10,
         "D": 100, "n_beta": 12, "site": 9},
        # a smaller active space, singlet, ragged, tensor cores
        {**hub, "name": "action_K10_D61_ab_initio_tc", "ham": "ab_initio", "K": 10, "N": 10, "twoM": 0, "twoS": 0,
         "D": 61, "n_beta": 6, "site": 3, "tc": True},
        # one two-site step on a shorter chain with the default options: Davidson's own kernels count
        {"name": "step_L16_D64", "kind": "step", "K": 16, "N": 16, "twoM": 0, "twoS": 0, "D": 64, "n_beta": 6,
         "site": 7, "U": 4.0, "form": "default", "settled": True},
        # the benchmark's step in the benchmark's fast form (3xTF32 until the residual is small, then FP64
        # products on the tensor cores, tuned tiles); like every solve it ends on the converged eigenvalue
        {"name": "step_L24_D256_fast", "kind": "step", "K": 24, "N": 24, "twoM": 0, "twoS": 0, "D": 256, "n_beta": 8,
         "site": 11, "U": 4.0, "form": "fast", "settled": True},
        # a full sweep without truncation, as the tests run it to the exact energy
        {"name": "sweep_L6_D64", "kind": "sweep", "K": 6, "N": 6, "twoM": 0, "twoS": 0, "D": 64, "n_beta": 4, "U": 4.0},
        # a random triplet state loaded, canonicalised and measured
        {"name": "load_L24_D256_S1", "kind": "load", "K": 24, "N": 24, "twoM": 2, "twoS": 2, "D": 256, "n_beta": 8,
         "U": 4.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _spins(rng, K, N, twoS_min=0):
    """2M and 2S of a random target of N electrons on K orbitals."""
    most = min(N, 2 * K - N, 4)
    start = twoS_min + (twoS_min + N) % 2
    twoS = rng.randrange(start, max(start, most) + 1, 2)
    return rng.randrange(-twoS, twoS + 1, 2), twoS


def draw(rng):
    kind = rng.choice(["action", "action", "action", "ab_initio", "step", "sweep", "load"])
    if kind in ("action", "ab_initio"):
        ab = kind == "ab_initio"
        K = _log(rng, 6, 14) if ab else _log(rng, 6, 24)
        N = max(2, min(2 * K - 2, K + rng.randrange(-K // 4, K // 4 + 1)))
        twoM, twoS = _spins(rng, K, N)
        return {"kind": "action", "ham": "ab_initio" if ab else "hubbard", "K": K, "N": N, "twoM": twoM, "twoS": twoS,
                "D": _log(rng, 12, 96) if ab else _log(rng, 12, 256), "n_beta": rng.randrange(2, 9),
                "site": rng.randrange(1, K - 2), "U": round(rng.uniform(1.0, 8.0), 2), "tc": rng.random() < 0.5, "settled": rng.random() < 0.5,
                "out": rng.choice(["yz", "yz", "y", "z"])}
    if kind == "step":
        # pairs near the middle, where the solve converges from a random state in some dozens of iterations
        K = rng.randrange(16, 25)
        return {"kind": "step", "K": K, "N": K, "twoM": K % 2, "twoS": K % 2, "D": _log(rng, 24, 256),
                "n_beta": (K + 3) // 3, "site": rng.randrange(K // 2 - 2, K // 2 + 1), "U": round(rng.uniform(2.0, 6.0), 2),
                "form": rng.choice(["default", "fast"]), "settled": rng.random() < 0.5}
    if kind == "sweep":
        K = rng.randrange(4, 7)
        twoS = K % 2 + 2 * rng.randrange(0, 2)
        return {"kind": "sweep", "K": K, "N": K, "twoM": twoS, "twoS": twoS, "D": 4 ** (K // 2), "n_beta": rng.randrange(4, 7),
                "U": round(rng.uniform(2.0, 6.0), 2)}
    K = _log(rng, 6, 24)
    N = max(2, K + rng.randrange(-2, 3))
    twoM, twoS = _spins(rng, K, N, 1)
    return {"kind": "load", "K": K, "N": N, "twoM": twoM, "twoS": twoS, "D": _log(rng, 16, 256),
            "n_beta": rng.randrange(4, 9), "U": round(rng.uniform(1.0, 8.0), 2)}


# ---- seeded states ------------------------------------------------------------------------------


def _structure(case):
    """Per bond the labels (n, 2m) -> dimension: in proportion to the smaller of the left and right Fock
    sectors (settled: to a bell around the mean filling and spin), at most D in all and at most that
    sector, labels without a neighbour on either side removed."""
    K, N, twoM, D = case["K"], case["N"], case["twoM"], case["D"]
    Na, Nb = (N + twoM) // 2, (N - twoM) // 2
    bonds = []
    for i in range(K + 1):
        w = {}
        for na in range(i + 1):
            for nb in range(i + 1):
                ra, rb = Na - na, Nb - nb
                if 0 <= ra <= K - i and 0 <= rb <= K - i:
                    w[(na + nb, na - nb)] = min(math.comb(i, na) * math.comb(i, nb), math.comb(K - i, ra) * math.comb(K - i, rb))
        total = sum(w.values())
        if total > D:
            room = w
            if case.get("settled"):
                w = {q: math.exp(-((q[0] - N * i / K) / 1.0) ** 2 / 2 - ((q[1] - twoM * i / K) / 1.9) ** 2 / 2) for q in w}
                total = sum(w.values())
            share = {q: min(D * v / total, room[q]) for q, v in w.items()}
            w = {q: int(s) for q, s in share.items()}
            for q in sorted(share, key=lambda q: (w[q] - share[q], q))[:D - sum(w.values())]:
                w[q] += w[q] < room[q]
        bonds.append({q: d for q, d in w.items() if d > 0})
    changed = True
    while changed:
        changed = False
        for i in range(K + 1):
            for q in list(bonds[i]):
                left = i == 0 or any((q[0] - _N[s], q[1] - _M[s]) in bonds[i - 1] for s in range(4))
                right = i == K or any((q[0] + _N[s], q[1] + _M[s]) in bonds[i + 1] for s in range(4))
                if not (left and right):
                    del bonds[i][q]
                    changed = True
    return bonds


def _limit_left(bonds, upto):
    for i in range(1, upto + 1):
        for q in bonds[i]:
            bonds[i][q] = min(bonds[i][q], sum(bonds[i - 1].get((q[0] - _N[s], q[1] - _M[s]), 0) for s in range(4)))


def _limit_right(bonds, downto):
    for i in range(len(bonds) - 2, downto - 1, -1):
        for q in bonds[i]:
            bonds[i][q] = min(bonds[i][q], sum(bonds[i + 1].get((q[0] + _N[s], q[1] + _M[s]), 0) for s in range(4)))


def _offsets(bond):
    off, at = {}, 0
    for q in sorted(bond):
        off[q] = at
        at += bond[q]
    return off, at


def _labels(bond):
    return np.array([q for q in sorted(bond) for _ in range(bond[q])], dtype=np.int64).reshape(-1, 2)


def _state(case, seed):
    """Labels per bond and dense (Dl, 4, Dr) site tensors.  With a centre: left-isometric left of it,
    right-isometric right of it, norm 1; without (kind load): Gaussian entries throughout."""
    K = case["K"]
    rng = np.random.default_rng(seed)
    bonds = _structure(case)
    centre = None if case["kind"] == "load" else case.get("site", 0)
    if centre is not None:
        _limit_left(bonds, centre)
        _limit_right(bonds, centre + 1)
    tensors = []
    for i in range(K):
        lo, nl = _offsets(bonds[i])
        ro, nr = _offsets(bonds[i + 1])
        A = np.zeros((nl, 4, nr))
        if centre is not None and i < centre:
            for q, d in bonds[i + 1].items():
                parts = [(s, (q[0] - _N[s], q[1] - _M[s])) for s in range(4)]
                parts = [(s, p, bonds[i][p]) for s, p in parts if p in bonds[i]]
                Q = np.linalg.qr(rng.standard_normal((sum(n for _, _, n in parts), d)))[0]
                at = 0
                for s, p, n in parts:
                    A[lo[p]:lo[p] + n, s, ro[q]:ro[q] + d] = Q[at:at + n]
                    at += n
        else:
            for p, d in bonds[i].items():
                parts = [(s, (p[0] + _N[s], p[1] + _M[s])) for s in range(4)]
                parts = [(s, q, bonds[i + 1][q]) for s, q in parts if q in bonds[i + 1]]
                width = sum(n for _, _, n in parts)
                if centre is not None and i > centre:
                    Q = np.linalg.qr(rng.standard_normal((width, d)))[0].T
                else:
                    Q = rng.standard_normal((d, width)) / math.sqrt(width)
                at = 0
                for s, q, n in parts:
                    A[lo[p]:lo[p] + d, s, ro[q]:ro[q] + n] = Q[:, at:at + n]
                    at += n
        if i == centre:
            A /= np.linalg.norm(A)
        tensors.append(A)
    return [_labels(b) for b in bonds], tensors


def _two_site_index(ql, qr):
    """Flat indices into the dense (Dl, 4, 4, Dr) tensor of the library's packed vector: per left label
    a row-major block of its rows, the columns over s = 4 s1 + s2 and the right indices allowed with it."""
    Dr, dense = qr.shape[0], []
    cols = {}
    for a in range(ql.shape[0]):
        q = (int(ql[a, 0]), int(ql[a, 1]))
        if q not in cols:
            cols[q] = np.concatenate([s * Dr + np.flatnonzero((qr[:, 0] == q[0] + _N[s >> 2] + _N[s & 3]) &
                                                              (qr[:, 1] == q[1] + _M[s >> 2] + _M[s & 3])) for s in range(16)])
        dense.append(a * 16 * Dr + cols[q])
    return np.concatenate(dense)


def _vector(case, seed, index):
    x = np.random.default_rng((seed, 1)).standard_normal(index.shape[0])
    return x / np.linalg.norm(x)


def _integrals(K, seed):
    """Active-space-like real integrals with the eightfold symmetry."""
    rng = np.random.default_rng((seed, 2))
    h1 = np.triu(rng.normal(0.0, 0.1, (K, K)), 1)
    h1 = h1 + h1.T + np.diag(rng.uniform(-3.0, -1.0, K))
    e = rng.normal(0.0, 0.02, (K, K, K, K))
    e = (e + e.transpose(1, 0, 2, 3)) / 2
    e = (e + e.transpose(0, 1, 3, 2)) / 2
    e = (e + e.transpose(2, 3, 0, 1)) / 2
    c = rng.uniform(0.3, 0.8, (K, K))
    c = np.triu(c) + np.triu(c, 1).T
    p = np.arange(K)
    e[p[:, None], p[:, None], p[None, :], p[None, :]] = c
    return h1, e


def _repulsion(case, seed):
    """U; another one for each seed of a sweep, whose result does not depend on the state it starts from."""
    return case["U"] * (np.random.default_rng((seed, 3)).uniform(0.9, 1.1) if case["kind"] == "sweep" else 1.0)


# ---- the framework's calls --------------------------------------------------------------------------


def _handle(case):
    from paper_1703_04789_gb300 import Spmps
    opts = {"fp64_tensor_cores": case.get("tc", False)}
    if case["kind"] == "step":
        opts = {"dav_max_iter": 600}
        if case["form"] == "fast":
            opts.update(precision="3xtf32", fp64_tensor_cores=True, autotune=True)
    return Spmps(case["K"], case["N"], case["twoM"], case["twoS"], case["n_beta"], case["D"], **opts)


def prepare(case, seed):
    dev = _handle(case)
    if case.get("ham") == "ab_initio":
        h1, h2 = _integrals(case["K"], seed)
        dev.set_hamiltonian(h1, h2, 0.0)
    else:
        dev.set_hubbard(1.0, _repulsion(case, seed))
    labels, tensors = _state(case, seed)
    state = {"case": case, "dev": dev, "labels": labels, "tensors": tensors}
    if case["kind"] == "action":
        k = case["site"]
        dev.set_mps(labels, tensors, center=k)
        x = torch.tensor(_vector(case, seed, _two_site_index(labels[k], labels[k + 2])), device="cuda")
        state["x"] = x
        state["y"] = torch.empty_like(x) if "y" in case["out"] else None
        state["z"] = torch.empty_like(x) if "z" in case["out"] else None
        # the environments and the plan of the pair, which an eigensolver's first call builds
        dev.apply_heff(k, x, state["y"], state["z"], stream=torch.cuda.current_stream())
    return state


def run(state):
    case, dev = state["case"], state["dev"]
    if case["kind"] == "action":
        dev.apply_heff(case["site"], state["x"], state["y"], state["z"], stream=torch.cuda.current_stream())
        return {o: state[o] for o in case["out"]}
    if case["kind"] == "load":
        dev.set_mps(state["labels"], state["tensors"], center=0)
        dev.canonicalize()
        energy, norm = dev.energy()
        return {"energy": energy, "norm": norm, "s2": dev.expect_s2()}
    # the new site tensors are defined up to their gauge and the kernel of the metric: the eigenvalue and the
    # energies are what two correct solves agree on
    dev.set_mps(state["labels"], state["tensors"], center=case.get("site", 0))
    if case["kind"] == "step":
        theta, _ = dev.optimize_step(case["site"], True, allow_not_converged=True)
        return {"theta": theta}
    energies, _ = dev.sweep(1)
    return {"energies": energies}


# ---- what a pass cannot do without -----------------------------------------------------------------


def _groups(bond):
    g = {}
    for (n, _), d in bond.items():
        g[n] = g.get(n, 0) + d
    return g


def _bonds(case):
    bonds = _structure(case)
    if case["kind"] != "load":
        _limit_left(bonds, case.get("site", 0))
        _limit_right(bonds, case.get("site", 0) + 1)
    return bonds


def _channels(case, k):
    """Channels of the operator at bond k by particle-number charge: the Hubbard chain's six, or those of
    the complementary-operator form (start, done, one or two operators on the smaller side)."""
    K = case["K"]
    if case.get("ham") != "ab_initio":
        return {0: 1} if k in (0, K) else {0: 2, 1: 2, -1: 2}
    nl, nr = 2 * k, 2 * (K - k)
    m = min(nl, nr)
    return {0: 2 + m * m, 1: nl + nr, -1: nl + nr, 2: m * (m - 1) // 2, -2: m * (m - 1) // 2}


def _action_work(case, k, out="yz"):
    """Both environments, x and the results once; the block products of the environments with x (phases A
    and C) and one multiply-add per element and channel for the operator between them."""
    bonds = _bonds(case)
    bl, br = bonds[k], bonds[k + 2]
    gl, gr, G = _groups(bl), _groups(br), case["n_beta"]
    flops = elements = 0
    nx = sum(d * br.get((q[0] + _N[s >> 2] + _N[s & 3], q[1] + _M[s >> 2] + _M[s & 3]), 0) for q, d in bl.items() for s in range(16))
    for chl, chr_, wanted in ((_channels(case, k), _channels(case, k + 2), "y" in out), ({0: 1}, {0: 1}, "z" in out)):
        if not wanted:
            continue
        for c, nw in chl.items():
            for n, rows in gl.items():
                if n - c not in gl:
                    continue
                elements += G * nw * rows * gl[n - c]
                for q, d in bl.items():
                    if q[0] == n - c:
                        w = sum(br.get((q[0] + _N[s >> 2] + _N[s & 3], q[1] + _M[s >> 2] + _M[s & 3]), 0) for s in range(16))
                        flops += 2 * G * nw * rows * d * w
        for c, nw in chr_.items():
            for n, cols in gr.items():
                if n - c not in gr:
                    continue
                elements += G * nw * cols * gr[n - c]
                for q, d in bl.items():
                    for s in range(16):
                        b = (q[0] + _N[s >> 2] + _N[s & 3], q[1] + _M[s >> 2] + _M[s & 3])
                        if b in br and b[0] == n:
                            flops += 2 * G * nw * d * br[b] * gr[n - c]
                flops += 2 * G * nw * gr[n - c] * sum(gl.get(n - _N[s >> 2] - _N[s & 3], 0) for s in range(16))
    return {"bytes": 8.0 * (elements + nx * (1 + len(out))), "flops": float(flops)}


def _state_elements(bonds):
    return sum(d * bonds[i + 1].get((q[0] + _N[s], q[1] + _M[s]), 0) for i in range(len(bonds) - 1) for q, d in bonds[i].items() for s in range(4))


def work(case):
    if case["kind"] == "action":
        return _action_work(case, case["site"], case["out"])
    K, bytes_, flops = case["K"], 8.0 * _state_elements(_bonds(case)), 0.0
    if case["kind"] == "step":
        w = _action_work(case, case["site"])
        return {"bytes": bytes_ + 50 * w["bytes"], "flops": 50 * w["flops"]}  # about fifty iterations
    # one action per pair for the environments on the way and the result (a sweep's solves: ten each)
    times = 10 * 2 if case["kind"] == "sweep" else 1
    for k in range(K - 1):
        w = _action_work(case, k)
        bytes_ += times * w["bytes"]
        flops += times * w["flops"]
    return {"bytes": bytes_, "flops": flops}


# ---- plain 64-bit references -------------------------------------------------------------------


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _quadrature(case):
    """Gauss-Legendre points in cos(beta) and c_g = (2S+1)/2 w_g d^S_MM(beta_g) (Wigner's sum)."""
    x, w = np.polynomial.legendre.leggauss(case["n_beta"])
    beta = np.arccos(x)
    p, m = (case["twoS"] + case["twoM"]) // 2, (case["twoS"] - case["twoM"]) // 2
    c, s = np.cos(beta / 2), np.sin(beta / 2)
    d = sum((-1) ** k * math.comb(p, k) * math.comb(m, k) * c ** (p + m - 2 * k) * s ** (2 * k) for k in range(min(p, m) + 1))
    return beta, 0.5 * (case["twoS"] + 1) * w * d


def _operator(case, which):
    """Dense MPO (K sites of (wl, wr, 4, 4)): the Hubbard chain, S^2, or the identity."""
    K = case["K"]
    one, z = np.eye(2), np.diag([1.0, -1.0])
    up = np.array([[0.0, 0.0], [1.0, 0.0]])
    ca, cb = np.kron(up, one), np.kron(z, up)
    par, eye = np.kron(z, z), np.eye(4)
    if which == "identity":
        return [eye.reshape(1, 1, 4, 4)] * K
    if which == "s2":
        plus = ca @ cb.T
        sz = 0.5 * (ca @ ca.T - cb @ cb.T)
        local = 0.5 * (plus @ plus.T + plus.T @ plus) + sz @ sz
        left, right = [plus, plus.T, 2 * sz], [plus.T, plus, sz]
    else:
        local = case["U"] * (ca @ ca.T @ cb @ cb.T)
        left, right = [ca @ par, cb @ par, par @ ca.T, par @ cb.T], [-ca.T, -cb.T, -ca, -cb]
    n = len(left) + 2
    W = np.zeros((n, n, 4, 4))
    W[0, 0] = W[n - 1, n - 1] = eye
    W[0, n - 1] = local
    for j, (a, b) in enumerate(zip(left, right)):
        W[0, j + 1], W[j + 1, n - 1] = a, b
        if which == "s2":
            W[j + 1, j + 1] = eye
    return [W[:1] if k == 0 else W[:, n - 1:] if k == K - 1 else W for k in range(K)]


def _rotated(mpo, beta, dev):
    """W r(beta) on the ket leg for every beta: K sites of (G, wl, wr, 4, 4)."""
    r = np.zeros((len(beta), 4, 4))
    c, s = np.cos(beta / 2), np.sin(beta / 2)
    r[:, 0, 0] = r[:, 3, 3] = 1.0
    r[:, 1, 1] = r[:, 2, 2] = c
    r[:, 1, 2], r[:, 2, 1] = s, -s
    return [torch.tensor(np.einsum("abst,gtu->gabsu", w, r), device=dev) for w in mpo]


def _left(L, A, W):
    t = torch.einsum("gwac,ctd->gwatd", L, A)
    t = torch.einsum("gwatd,gwvst->gvasd", t, W)
    return torch.einsum("gvasd,asb->gvbd", t, A)


def _environments(A, W, k, G):
    L = torch.ones(G, 1, 1, 1, dtype=torch.float64, device=A[0].device)
    R = L.clone()
    for i in range(k):
        L = _left(L, A[i], W[i])
    for i in range(len(A) - 1, k + 1, -1):
        R = _left(R, A[i].permute(2, 1, 0), W[i].transpose(1, 2))
    return L, R


def _apply(L, R, W1, W2, c, x):
    y = torch.zeros_like(x)
    for g in range(len(c)):
        t = torch.einsum("wac,ctud->watud", L[g], x)
        t = torch.einsum("watud,wvst->vasud", t, W1[g])
        t = torch.einsum("vasud,vwpu->waspd", t, W2[g])
        y += c[g] * torch.einsum("waspd,wbd->aspb", t, R[g])
    return y


def exact(case, seed):
    dev = _device()
    if case["kind"] == "sweep":
        # the chain's lowest energy with 2M = 2S (its spin grows with |M|: Lieb and Mattis), dense
        K, blocks = case["K"], []
        for n in ((case["N"] + case["twoM"]) // 2, (case["N"] - case["twoM"]) // 2):
            masks = [b for b in range(1 << K) if bin(b).count("1") == n]
            at = {b: i for i, b in enumerate(masks)}
            T = np.zeros((len(masks), len(masks)))
            for b in masks:
                for p in range(K - 1):
                    if (b >> p) & 1 != (b >> (p + 1)) & 1:
                        T[at[b ^ (3 << p)], at[b]] = -1.0
            blocks.append((masks, T))
        (ma, Ta), (mb, Tb) = blocks
        H = np.kron(Ta, np.eye(len(mb))) + np.kron(np.eye(len(ma)), Tb)
        H += np.diag([_repulsion(case, seed) * bin(a & b).count("1") for a in ma for b in mb])
        return {"energies": np.linalg.eigvalsh(H)[:1]}
    if case["kind"] == "step":
        return None  # a dense generalised eigenproblem of up to 66 thousand unknowns: far over twenty seconds
    beta, c = _quadrature(case)
    labels, tensors = _state(case, seed)
    A = [torch.tensor(t, device=dev) for t in tensors]
    if case["kind"] == "action":
        k = case["site"]
        index = torch.tensor(_two_site_index(labels[k], labels[k + 2]), device=dev)
        x = torch.zeros(A[k].shape[0], 4, 4, A[k + 1].shape[2], dtype=torch.float64, device=dev)
        x.view(-1)[index] = torch.tensor(_vector(case, seed, index), device=dev)
        out = {}
        for o in case["out"]:
            if o == "y" and case["ham"] == "ab_initio":
                out[o] = None  # a dense operator of hundreds of channels: far over twenty seconds
                continue
            W = _rotated(_operator(case, "hubbard" if o == "y" else "identity"), beta, dev)
            L, R = _environments(A, W, k, len(beta))
            out[o] = _apply(L, R, W[k], W[k + 1], c, x).reshape(-1)[index].cpu()
        return out
    values = {}
    for which in ("hubbard", "s2", "identity"):
        W = _rotated(_operator(case, which), beta, dev)
        L = torch.ones(len(beta), 1, 1, 1, dtype=torch.float64, device=dev)
        for i in range(case["K"]):
            L = _left(L, A[i], W[i])
        values[which] = float((torch.tensor(c, device=dev) * L.reshape(-1)).sum())
    L = torch.ones(1, 1, 1, 1, dtype=torch.float64, device=dev)
    for a, w in zip(A, _rotated(_operator(case, "identity"), np.zeros(1), dev)):
        L = _left(L, a, w)
    return {"energy": values["hubbard"] / values["identity"], "norm": values["identity"] / float(L), "s2": values["s2"] / values["identity"]}
