"""The work a user of this library has it do, as measurable cases.

Every case goes through the package's public entry points (``from_model``,
``ttn_step``, ``ttn_batch_step``, ``ttn_rdm``, ``ttn_get_node``). The models
are the ones of the repository's own configurations and tests -- the
spin-boson tensor train, the Table 1 spin-boson, the Frenkel exciton chain,
the three-site FMO model, batches of uneven spin-boson instances, the driven
structured two-level system -- with their sizes; bath and site parameters and
the state are drawn from the seed.

The state is a generic point of the manifold: the product state every
propagation starts from plus random components on every direction, smaller
towards high Fock levels and high bond indices, as a propagation under way has
them. (From the bare product state most directions carry no weight at all, so
their tensors say nothing about what was computed.)

A propagation pass is a chunk of steps, then rho_S and the state read back,
which is what a program that records a trajectory and keeps restart data does.
An adaptive-rank run's node tensors are defined up to the phases of the
singular vectors, so that case reads rho_S and the ranks.
"""
from __future__ import annotations

import dataclasses
import math
from typing import List, Optional, Tuple

import numpy as np

import paper_2603_17711_gb300 as pkg

CM1 = 2.0 * np.pi * 2.99792458e10 * 1e-15  # 1 cm^-1 in rad/fs
KB = 0.6950348                             # cm^-1 per kelvin
SX = np.array([[0, 1], [1, 0]], np.complex128)
SZ = np.diag([1.0, -1.0]).astype(np.complex128)
FMO_H = np.array([[200.0, -87.7, 5.5], [-87.7, 320.0, 30.8], [5.5, 30.8, 0.0]])
FMO_BO = [(26.24, 160.0, 133.0), (13.832, 247.0, 53.0), (101.479, 763.0, 76.0),
          (57.575, 1175.0, 29.0), (25.764, 1356.0, 29.0), (9.126, 1521.0, 15.0)]


@dataclasses.dataclass
class Bath:
    Q: np.ndarray
    beta: float
    dl: Optional[Tuple[float, float]] = None
    bo: List[Tuple[float, float, float]] = dataclasses.field(default_factory=list)
    n_ltc: int = 0
    scheme: str = "pade"

    @property
    def n_features(self) -> int:
        return (1 if self.dl else 0) + 2 * len(self.bo) + self.n_ltc


@dataclasses.dataclass
class Drive:
    V: np.ndarray
    amp: float
    omega: float

    def g(self, t: float) -> float:
        return self.amp * math.cos(self.omega * t)

    @property
    def bound(self) -> float:
        return abs(self.amp)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # rho_S read between steps: the smallest call, made after every step of a recorded trajectory
        dict(name="read_rdm_chain", op="rdm", model="chain", n=7, depth=8, rank=20, ltc=2),
        # the plain spin-boson tensor train: the smallest propagation, bound by latency and launches
        dict(name="sb_train_r10", op="ps1", model="sb", tree="tt", ltc=3, depth=10, rank=10, mixed=False, steps=8),
        # the same family at an odd rank and depth, a feature count that does not divide
        dict(name="sb_tree_r19_odd", op="ps1", model="sb", tree="btt", ltc=4, depth=11, rank=19, mixed=False, steps=6),
        # the paper's Table 1 spin-boson: a deep hierarchy on a small tree
        dict(name="sb_table1_r20", op="ps1", model="sb_table1", depth=25, rank=20, ltc=1, mixed=False, steps=4),
        # the seven-site exciton chain at rank 20: the ordinary propagation, in both precisions
        dict(name="chain_r20", op="ps1", model="chain", n=7, depth=8, rank=20, ltc=2, mixed=False, steps=2),
        dict(name="chain_r20_mixed", op="ps1", model="chain", n=7, depth=8, rank=20, ltc=2, mixed=True, steps=2),
        # three-site FMO with six Brownian peaks: many features, many small nodes
        dict(name="fmo_r16", op="ps1", model="fmo", depth=20, rank=16, ltc=3, mixed=False, steps=1),
        # the chain at rank 64: the largest states, in both precisions
        dict(name="chain_r64", op="ps1", model="chain", n=7, depth=8, rank=64, ltc=2, mixed=False, steps=1),
        dict(name="chain_r64_mixed", op="ps1", model="chain", n=7, depth=8, rank=64, ltc=2, mixed=True, steps=2),
        # many uneven spin-boson instances advanced together
        dict(name="batch_sb_64", op="batch", model="sb_batch", count=64, steps=1),
        # adaptive rank under a drive: two-site updates and their singular value decompositions
        dict(name="driven_ps2_cap16", op="ps2", model="tls", depth=10, rank=16, ltc=1, steps=1),
        # direct integration of all nodes together
        dict(name="chain_vmf_r12", op="vmf", model="chain", n=4, depth=6, rank=12, ltc=2, steps=1),
    ]


def _logint(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = work(next(c for c in listed() if c["name"] == "chain_r64"))["flops"]
    while True:
        kind = rng.choice(["rdm", "sb", "sb", "sb_table1", "chain", "chain", "chain", "fmo", "batch", "ps2", "vmf"])
        if kind == "rdm":
            c = dict(op="rdm", model="chain", n=rng.randint(3, 7), depth=rng.randint(4, 9), rank=_logint(rng, 10, 48),
                     ltc=rng.randint(1, 3))
        elif kind == "sb":
            c = dict(op="ps1", model="sb", tree=rng.choice(["tt", "btt"]), ltc=rng.randint(2, 4),
                     depth=rng.randint(6, 12), rank=_logint(rng, 8, 40), mixed=rng.random() < 0.3,
                     steps=rng.randint(2, 6))
        elif kind == "sb_table1":
            c = dict(op="ps1", model="sb_table1", depth=rng.randint(12, 25), rank=_logint(rng, 10, 40), ltc=1,
                     mixed=False, steps=rng.randint(1, 4))
        elif kind == "chain":
            c = dict(op="ps1", model="chain", n=rng.randint(4, 7), depth=rng.randint(5, 8), rank=_logint(rng, 12, 64),
                     ltc=2, mixed=rng.random() < 0.4, steps=1)
        elif kind == "fmo":
            c = dict(op="ps1", model="fmo", depth=rng.randint(12, 20), rank=_logint(rng, 10, 24), ltc=rng.randint(1, 3),
                     mixed=rng.random() < 0.3, steps=1)
        elif kind == "batch":
            c = dict(op="batch", model="sb_batch", count=_logint(rng, 8, 64), steps=1)
        elif kind == "ps2":
            c = dict(op="ps2", model="tls", depth=rng.randint(6, 10), rank=_logint(rng, 8, 18), ltc=rng.randint(0, 2),
                     steps=1)
        else:
            c = dict(op="vmf", model="chain", n=rng.randint(3, 5), depth=rng.randint(5, 8), rank=_logint(rng, 8, 20),
                     ltc=rng.randint(1, 2), steps=1)
        if work(c)["flops"] <= top:
            return c


# ---------------------------------------------------------------------------
# models
# ---------------------------------------------------------------------------

@dataclasses.dataclass
class Model:
    H: np.ndarray
    baths: list
    depth: List[int]
    parent: List[int]
    leg_node: List[int]
    ranks: List[int]
    dt: float
    drives: list = dataclasses.field(default_factory=list)

    @property
    def leg_dims(self) -> List[int]:
        return [self.H.shape[0]] * 2 + list(self.depth)


def _train(K: int):
    if K == 1:
        return [-1], [0, 0, 0]
    return [-1] + list(range(K - 1)), [0, 0] + [min(k + 1, K - 1) for k in range(K)]


def _binary(K: int):
    parent, leg_node = [-1], [0, 0] + [-1] * K
    if K == 1:
        return parent, [0, 0, 0]

    def build(lo, hi, par):
        n = hi - lo
        if n == 1:
            leg_node[2 + lo] = par
            return
        u = len(parent)
        parent.append(par)
        if n == 2:
            leg_node[2 + lo] = leg_node[3 + lo] = u
            return
        mid = lo + (n + 1) // 2
        build(lo, mid, u)
        build(mid, hi, u)

    build(0, K, 0)
    return parent, leg_node


def _model(case, rng) -> Model:
    kind = case["model"]
    drives = []
    if kind == "sb":
        H = rng.uniform(0.4, 0.6) * SZ + rng.uniform(0.9, 1.1) * SX
        baths = [Bath(SZ, 1.0, dl=(rng.uniform(0.45, 0.5), rng.uniform(0.95, 1.0)), n_ltc=case["ltc"])]
        dt = 0.01
    elif kind == "sb_table1":
        H = (np.array([[-750.0, 300.0], [300.0, 750.0]]) * rng.uniform(0.98, 1.0)).astype(np.complex128) * CM1
        baths = [Bath(np.diag([-0.5, 0.5]).astype(np.complex128), 1.0 / (KB * 300.0 * CM1),
                      dl=(rng.uniform(520.0, 540.0) * CM1, 70.0 * CM1), bo=[(161.6 * CM1, 1243.0 * CM1, 10.0 * CM1)],
                      n_ltc=case["ltc"])]
        dt = 1.0
    elif kind == "chain":
        n = case["n"]
        H = np.diag(rng.normal(0.0, 100.0, n)).astype(np.complex128)
        for i, v in enumerate(rng.uniform(50.0, 100.0, n - 1)):
            H[i, i + 1] = H[i + 1, i] = v
        H = H * CM1
        baths = []
        for b in range(n):
            Q = np.zeros((n, n), np.complex128)
            Q[b, b] = 1.0
            baths.append(Bath(Q, 1.0 / (KB * 300.0 * CM1), dl=(35.0 * CM1, 106.0 * CM1), n_ltc=case["ltc"]))
        dt = 0.02 if case["op"] == "vmf" else 0.05
    elif kind == "fmo":
        H = (FMO_H + np.diag(rng.uniform(-10.0, 10.0, 3))).astype(np.complex128) * CM1
        baths = []
        for b in range(3):
            Q = np.zeros((3, 3), np.complex128)
            Q[b, b] = 1.0
            baths.append(Bath(Q, 1.0 / (KB * 77.0 * CM1), bo=[tuple(x * CM1 for x in p) for p in FMO_BO],
                              n_ltc=case["ltc"]))
        dt = 0.05
    elif kind == "tls":
        H = rng.uniform(0.7, 0.8) * SZ
        baths = [Bath(SZ, 1.0, dl=(0.2, 1.0), bo=[(0.1, 1.0, 0.1), (0.1, 2.0, 0.1), (0.1, 3.0, 0.1)],
                      n_ltc=case["ltc"])]
        drives = [Drive(SX, 0.2, 1.5)]
        dt = 0.01
    else:
        raise ValueError(kind)
    K = sum(b.n_features for b in baths)
    parent, leg_node = _train(K) if case.get("tree") == "tt" else _binary(K)
    return Model(H, baths, [case["depth"]] * K, parent, leg_node, [0] + [case["rank"]] * (len(parent) - 1), dt, drives)


def _batch_models(case, rng) -> List[Model]:
    """Uneven spin-boson instances: sizes from a fixed sequence (the same for every
    seed, so that the work is), bath and system parameters from the seed, where
    the truncated hierarchies are stable."""
    sizes = np.random.default_rng(4242)
    out = []
    for _ in range(case["count"]):
        K, depth, rank = int(sizes.integers(2, 9)), int(sizes.integers(6, 13)), int(sizes.integers(8, 33))
        H = 0.5 * rng.uniform(0.0, 2.0) * SZ + rng.uniform(0.0, 2.0) * SX
        bath = Bath(SZ, rng.uniform(4.0, 5.0), dl=(rng.uniform(0.1, 0.3), rng.uniform(0.5, 0.8)), n_ltc=K - 1)
        parent, leg_node = _binary(K)
        out.append(Model(H, [bath], [depth] * K, parent, leg_node, [0] + [rank] * (len(parent) - 1), 0.01))
    return out


# ---------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------

def _legs(m: Model):
    """Canonical legs of every node: parent bond first, then child nodes and open
    legs by the smallest open leg below them; ('p'|'n'|'o', index)."""
    n = len(m.parent)
    low = [10 ** 9] * n
    for leg, u in enumerate(m.leg_node):
        while u >= 0:
            low[u] = min(low[u], leg)
            u = m.parent[u]
    out = []
    for u in range(n):
        rest = [(low[c], "n", c) for c in range(n) if m.parent[c] == u]
        rest += [(leg, "o", leg) for leg, w in enumerate(m.leg_node) if w == u]
        out.append(([("p", u)] if u else []) + [(k, v) for _, k, v in sorted(rest)])
    return out


def _node_dims(m: Model):
    """Three leg dimensions of every node at the effective ranks: each bond capped
    by the product of the other legs at either end, to a fixed point."""
    legs, r = _legs(m), list(m.ranks)
    dim = lambda k, v: m.leg_dims[v] if k == "o" else r[v]  # noqa: E731
    while True:
        old = list(r)
        for u in range(1, len(r)):
            for w, own in ((u, ("p", u)), (m.parent[u], ("n", u))):
                r[u] = min(r[u], math.prod(dim(k, v) for k, v in legs[w] if (k, v) != own))
        if r == old:
            return [tuple(dim(k, v) for k, v in ls) for ls in legs], r


def _generic_state(dims, rng):
    nodes = []
    for u, d in enumerate(dims):
        fall = np.ones(d)
        for ax, n in enumerate(d):
            shape = [1, 1, 1]
            shape[ax] = n
            if u or ax == 2:
                fall = fall * np.exp(-2.0 * np.arange(n) / n).reshape(shape)
        G = (rng.normal(size=d) + 1j * rng.normal(size=d)) * fall
        if u == 0:
            A = 0.1 * G / math.sqrt(G.size)
            M = d[0]
            X = rng.normal(size=(M, M)) + 1j * rng.normal(size=(M, M))
            rho = X @ X.conj().T
            A[:, :, 0] += rho / np.trace(rho).real
            nodes.append(A)
        else:
            r, cols = d[0], d[1] * d[2]
            E = np.eye(r, cols, dtype=np.complex128) + 0.5 * G.reshape(r, cols) / math.sqrt(cols)
            q, t = np.linalg.qr(E.conj().T)
            ph = np.diag(t) / np.abs(np.diag(t))
            nodes.append(np.ascontiguousarray((q * ph).conj().T).reshape(d))
    return nodes


def _handle(m: Model, rng, precision=pkg.TTN_FP64, params=None):
    t = pkg.from_model(m.H, m.baths, m.depth, m.parent, m.leg_node, m.ranks, drives=m.drives, precision=precision,
                       params=params)
    dims = [t.ttn_node_shape(u) for u in range(t.n_nodes)]
    for u, T in enumerate(_generic_state(dims, rng)):
        t.ttn_set_node(u, T)
    return t


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["op"] == "batch":
        # instances that fill the GPU together: one CTA per tile, four warps each
        models = _batch_models(case, rng)
        return dict(case=case, dt=0.01, hs=[_handle(m, rng, params=dict(max_split=1, tile_warps=4)) for m in models])
    m = _model(case, rng)
    params = dict(max_rank=case["rank"], ps2_atol=1e-6, ps2_ratio=2.0) if case["op"] == "ps2" else None
    precision = pkg.TTN_MIXED_FP32 if case.get("mixed") else pkg.TTN_FP64
    return dict(case=case, dt=m.dt, h=_handle(m, rng, precision, params))


def run(state):
    case, dt = state["case"], state["dt"]
    op = case["op"]
    if op == "rdm":
        return state["h"].ttn_rdm()
    if op == "batch":
        hs = state["hs"]
        pkg.ttn_batch_step(hs, dt, pkg.TTN_PS1, case["steps"])
        rho = np.stack([h.ttn_rdm() for h in hs])
        nodes = [np.concatenate([h.ttn_get_node(u).reshape(-1) for u in range(h.n_nodes)]) for h in hs]
        return dict(rho=rho, state=np.concatenate(nodes))
    h = state["h"]
    if op == "ps2":
        h.ttn_step(dt, pkg.TTN_PS2, case["steps"])
        return dict(rho=h.ttn_rdm(), ranks=h.ttn_get_ranks())
    h.ttn_step(dt, pkg.TTN_VMF if op == "vmf" else pkg.TTN_PS1, case["steps"])
    return dict(rho=h.ttn_rdm(), nodes=[h.ttn_get_node(u) for u in range(h.n_nodes)])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _step_flops(m: Model, nodes_per_step=2, kappa=2.5):
    """FLOPs of one ps1 step: RK4 node and bond flows with the terms of a bath
    merged behind its coupling operator, the environments, the gauge moves
    (Householder QR with explicit Q) and the absorbed bond matrices; complex
    multiply-add = 8."""
    dims, r = _node_dims(m)
    legs = _legs(m)
    n = len(m.parent)
    bath_of = {}
    leg = 2
    for b, bath in enumerate(m.baths):
        for _ in range(bath.n_features):
            bath_of[leg] = b
            leg += 1
    below = [set() for _ in range(n)]
    for l_, u in enumerate(m.leg_node):
        while u >= 0:
            if l_ in bath_of:
                below[u].add(bath_of[l_])
            u = m.parent[u]
    arr = pkg.heom.heom_sop(m.H, m.baths, m.depth, m.drives)
    off, data = arr["op_offset"], arr["op_data"].view(np.complex128)
    norms = []
    for k, l_ in enumerate(arr["op_leg"]):
        d = m.leg_dims[l_]
        norms.append(np.linalg.norm(data[off[k]:off[k] + d * d].reshape(d, d), 2))
    lam = 0.0
    to = arr["term_offsets"]
    for t in range(len(to) - 1):
        c = abs(complex(arr["coef"][2 * t], arr["coef"][2 * t + 1]))
        c *= 1.0 if arr["coef_drive"][t] < 0 else m.drives[arr["coef_drive"][t]].bound
        lam += c * math.prod(norms[i] for i in arr["term_ops"][to[t]:to[t + 1]])
    sub = lambda tau: max(1, math.ceil(tau * lam / kappa - 1e-9))  # noqa: E731

    def keys(k, v):  # baths with a feature behind this lower leg
        return below[v] if k == "n" else ({bath_of[v]} if v in bath_of else set())

    total = 0.0
    for u in range(n):
        P = math.prod(dims[u])
        app = sum(8.0 * P * d for d in dims[u])  # single-leg sums
        for i, (k, v) in enumerate(legs[u]):
            if k == "p" or (k == "o" and v < 2):
                continue
            app += 2 * len(keys(k, v)) * 8.0 * P * dims[u][i]  # partners of Q and of its conjugate
        if u:
            app += 2 * len(below[u]) * 8.0 * P * dims[u][0]
        else:
            app += sum(len(m.baths) * 8.0 * P * d for d in dims[0][:2])
        total += (4 * sub(m.dt) if u == 0 else 2 * 4 * sub(0.5 * m.dt)) * app
    for u in range(1, n):
        d, nb = r[u], 2 * len(below[u])
        total += 2 * 4 * sub(0.5 * m.dt) * 8.0 * d ** 3 * (2 + 2 * nb)       # bond flow
        for w in (u, m.parent[u]):
            P = math.prod(dims[w])
            total += 2 * 8.0 * P * sum(dims[w])                              # environments: classes and projection
            total += 2 * 2 * 8.0 * P * d * max(1, nb)
            total += 2 * 16.0 * (2.0 * P * d - 2.0 * d ** 3 / 3.0)           # QR
            total += 2 * 8.0 * P * d                                         # absorbed bond matrix
    return total


def work(case):
    rng = np.random.default_rng(0)
    if case["op"] == "batch":
        ms = _batch_models(case, rng)
        state = sum(math.prod(d) for m in ms for d in _node_dims(m)[0])
        return dict(bytes=2 * 16.0 * state, flops=case["steps"] * sum(_step_flops(m) for m in ms))
    m = _model(case, rng)
    dims, r = _node_dims(m)
    state = sum(math.prod(d) for d in dims)
    if case["op"] == "rdm":
        M = m.H.shape[0]
        return dict(bytes=16.0 * (state + M * M), flops=8.0 * state)
    flops = _step_flops(m)
    if case["op"] == "vmf":  # seven right-hand sides, each a node application and the environments: about as many
        flops *= 7.0 / 8.0
    if case["op"] == "ps2":  # the two-site flows and the singular value decompositions of the merged pairs
        for u in range(1, len(r)):
            a = math.prod(dims[u]) / r[u]
            b = math.prod(dims[m.parent[u]]) / r[u]
            k, big = min(a, b), max(a, b)
            flops += 2 * 8.0 * (4 * a * b * sum(dims[u] + dims[m.parent[u]]) + 2 * big * k * k + 11 * k ** 3)
    return dict(bytes=2 * 16.0 * state, flops=case["steps"] * flops)


# ---------------------------------------------------------------------------
# 64-bit reference
# ---------------------------------------------------------------------------

def exact(case, seed):
    """rho_S of the prepared state: every feature leg contracted with its n = 0
    vector. A step has no short 64-bit statement of its own."""
    if case["op"] != "rdm":
        return None
    rng = np.random.default_rng(seed)
    m = _model(case, rng)
    dims, _ = _node_dims(m)
    nodes, legs = _generic_state(dims, rng), _legs(m)
    vec = [None] * len(nodes)
    for u in reversed(range(1, len(nodes))):  # children have higher numbers than their parents
        T = nodes[u]
        for k, v in reversed(legs[u][1:]):
            T = T[..., 0] if k == "o" else T @ vec[v]
        vec[u] = T
    k, v = legs[0][2]
    return nodes[0][:, :, 0] if k == "o" else nodes[0] @ vec[v]
