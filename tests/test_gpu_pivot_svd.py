"""The two-site split by pivoted QR and Jacobi on R^H (smaller side above 32
columns): one adaptive-rank step from a generic state against the oracle's
LAPACK split, at sizes where the blocking can go wrong (33 columns, odd counts,
more isometry columns than CTAs, a numerically rank-deficient matrix), and a
non-finite state.

Tolerance: both sides split the same matrix to 1e-14 of its norm and keep the
same number of singular triplets; what differs is rounding, amplified by the
gaps kept in the truncation (1e-4): 1e-10 on rho_S, equal ranks."""
import numpy as np
import pytest

import workloads as W
from oracle import ttn as ottn
from test_gpu_exact_split import generic_nodes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2603_17711_gb300 as p
    p.library()
    return p


def pair(pkg, depth, rank, n_pade, generic, ratio=2.0):
    w = W.driven_structured_tls(n_steps=1, n_pade=n_pade, depth=depth, cap=rank)
    w.ranks = W.uniform_ranks(w.parent, rank if generic else 4)
    g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, drives=w.drives,
                       params=dict(max_rank=rank, ps2_atol=1e-6, ps2_ratio=ratio))
    o = ottn.from_workload(w, params=ottn.Params(max_rank=rank, ps2_atol=1e-6, ps2_ratio=ratio))
    if generic:
        nodes = generic_nodes([g.ttn_node_shape(u) for u in range(g.n_nodes)], np.random.default_rng(11))
        for u, T in enumerate(nodes):
            g.ttn_set_node(u, T)
        o.tensors = [n.copy() for n in nodes]
        for c in o.tree.postorder():
            if c != 0:
                o.update_env(c, o.tree.parent[c])
    return w, g, o


@pytest.mark.parametrize("depth,rank,n_pade,generic", [
    (6, 6, 0, True),     # 36 columns: just above the cluster kernel
    (7, 11, 1, True),    # 49 / 77 / 121 columns, odd
    (10, 16, 1, True),   # 100 x 256
    (10, 16, 1, False),  # from the product state: numerically rank deficient
])
def test_step_matches_the_oracle(pkg, depth, rank, n_pade, generic):
    w, g, o = pair(pkg, depth, rank, n_pade, generic)
    for _ in range(1 if generic else 4):
        g.ttn_step(w.dt, pkg.TTN_PS2, 1)
        o.step(w.dt, "ps2")
    assert list(g.ttn_get_ranks()) == list(o.ranks)
    assert np.max(np.abs(g.ttn_rdm() - o.rdm())) <= 1e-10
    for u in range(1, g.n_nodes):  # every isometry semi-unitary toward the root
        T = g.ttn_get_node(u)
        A = T.reshape(T.shape[0], -1)
        assert np.max(np.abs(A @ A.conj().T - np.eye(T.shape[0]))) <= 1e-12, u
    g.close()


def test_non_finite_state_is_reported(pkg):
    w, g, o = pair(pkg, 7, 11, 1, True)
    big = g.ttn_get_node(0)
    g.ttn_set_node(0, big * (1e308 / np.max(np.abs(big))))
    with pytest.raises(pkg.TTNError):
        g.ttn_step(w.dt, pkg.TTN_PS2, 1)
        g.ttn_rdm()
    g.close()
