"""FP64 contractions on the tensor cores by the exact digit split: one step from
a generic state against the oracle at the sizes where the blocking can go wrong
(leg dimensions at and beside the 8-row blocks and the 64 limit, a leg above it
that has to stay on the CUDA cores), invariance under powers of two, and the
report of non-finite amplitudes.

Tolerance: a step applies a few hundred contractions, each within 1e-15 of the
exact sum relative to its operands (the digits lose less than the FP64 chain),
on nodes of unit norm: 1e-11 on the node tensors leaves two orders."""
import numpy as np
import pytest

import workloads as W
from oracle import ttn as ottn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2603_17711_gb300 as p
    p.library()
    return p


def generic_nodes(shapes, rng):
    """Random semi-unitary nodes near the product state, a full root."""
    out = []
    for u, d in enumerate(shapes):
        G = rng.normal(size=d) + 1j * rng.normal(size=d)
        if u == 0:
            A = 0.1 * G / np.sqrt(G.size)
            A[0, 0, 0] += 1.0
            out.append(A)
            continue
        r, cols = d[0], d[1] * d[2]
        E = np.eye(r, cols, dtype=np.complex128) + 0.5 * G.reshape(r, cols) / np.sqrt(cols)
        q, t = np.linalg.qr(E.conj().T)
        ph = np.diag(t) / np.abs(np.diag(t))
        out.append(np.ascontiguousarray((q * ph).conj().T).reshape(d))
    return out


def handle(pkg, w, nodes=None, **kw):
    g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, **kw)
    if nodes is None:
        nodes = generic_nodes([g.ttn_node_shape(u) for u in range(g.n_nodes)], np.random.default_rng(3))
    for u, T in enumerate(nodes):
        g.ttn_set_node(u, T)
    return g, nodes


def split_work(g):
    """Largest possible FLOPs of one contraction list (dims, terms of the tuning rows)."""
    r = g.ttn_tuning_get()
    r = r[r[:, 0] == 0].astype(float)
    return np.max(8.0 * r[:, 2] * r[:, 3] * r[:, 4] * r[:, 5] * np.max(r[:, 2:6], axis=1) * r[:, 7] * r[:, 6])


CASES = [
    ("chain", dict(n_sites=2, rank=64, depth=8)),   # 64: the largest leg, full blocks
    ("chain", dict(n_sites=2, rank=63, depth=9)),   # one short of full blocks, nine = one row over
    ("chain", dict(n_sites=2, rank=66, depth=9)),   # above the limit: those legs stay on the CUDA cores
    ("chain", dict(n_sites=2, rank=41, depth=7)),   # five row blocks: idle warps in the CTA
    ("chain", dict(n_sites=3, rank=25, depth=5)),   # 16-position tiles with a remainder
    ("train", dict(rank=33, depth=17)),             # tensor train: open legs in the middle
    ("train", dict(rank=16, depth=24)),             # whole blocks on every leg
]


@pytest.mark.parametrize("kind,args", CASES)
def test_step_matches_the_oracle(pkg, kind, args):
    w = W.exciton_chain(**args) if kind == "chain" else W.spin_boson_tt(n_pade=2, **args)
    g, nodes = handle(pkg, w)
    assert split_work(g) >= 8e6  # the list sizes that take the digit split
    o = ottn.from_workload(w)
    o.tensors = [n.copy() for n in nodes]
    for c in o.tree.postorder():
        if c != 0:
            o.update_env(c, o.tree.parent[c])
    g.ttn_step(w.dt, pkg.TTN_PS1, 1)
    o.step(w.dt, "ps1")
    assert np.max(np.abs(g.ttn_rdm() - o.rdm())) <= 1e-11
    for u in range(g.n_nodes):
        assert np.max(np.abs(g.ttn_get_node(u) - o.tensors[u])) <= 1e-11, u
    g.close()


def test_power_of_two_scaling_is_exact(pkg):
    """The equations are linear in the root's weight and every scale of the split
    is a power of two: the step of 2^40 x the state is 2^40 x the step, bit for bit."""
    w = W.exciton_chain(n_sites=2, rank=40, depth=8)
    g, nodes = handle(pkg, w)
    g.ttn_step(w.dt, pkg.TTN_PS1, 1)
    a = g.ttn_get_node(0)
    g.close()
    h, _ = handle(pkg, w, [nodes[0] * 2.0 ** 40] + nodes[1:])
    h.ttn_step(w.dt, pkg.TTN_PS1, 1)
    assert np.array_equal(h.ttn_get_node(0), a * 2.0 ** 40)
    h.close()


def test_overflow_is_reported(pkg):
    """Amplitudes that overflow inside the contractions still reach the finiteness check."""
    w = W.exciton_chain(n_sites=2, rank=40, depth=8)
    g, nodes = handle(pkg, w)
    g.ttn_set_node(0, nodes[0] * (1e308 / np.max(np.abs(nodes[0]))))
    g.ttn_step(1e4 * w.dt, pkg.TTN_PS1, 1)
    with pytest.raises(pkg.TTNError):
        g.ttn_rdm()
    g.close()
