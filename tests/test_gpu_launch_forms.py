"""The forms a launch takes by its size: operators with at most three diagonals
(legs above 12), pair products shared by lists, job tables in parameters or in
memory, the cluster QR with its Gram and solves in shared or in global memory, the
density matrix by tree levels, and the direct integration's inverse in shared or
in global memory. One step from a generic state against the oracle.

Tolerance: as for any step, a few hundred contractions within 1e-15 of the
exact sums on nodes of unit norm: 1e-11. Direct integration: the inverse of a
density matrix regularised by 1e-3 amplifies that a thousandfold at most, and
the step sizes agree to the same digits: 1e-10."""
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


def pair(pkg, w, params=None):
    g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, drives=w.drives,
                       params=params or {})
    o = ottn.from_workload(w, **({"params": ottn.Params(**params)} if params else {}))
    nodes = generic_nodes([g.ttn_node_shape(u) for u in range(g.n_nodes)], np.random.default_rng(5))
    for u, T in enumerate(nodes):
        g.ttn_set_node(u, T)
    o.tensors = [n.copy() for n in nodes]
    for c in o.tree.postorder():
        if c != 0:
            o.update_env(c, o.tree.parent[c])
    return g, o


def driven(depth):
    w = W.driven_structured_tls(n_pade=1, depth=depth)
    w.ranks = W.uniform_ranks(w.parent, 5)
    return w


STEPS = [
    lambda: W.spin_boson_tt(rank=5, depth=12, n_pade=2),              # the last dense leg
    lambda: W.spin_boson_tt(rank=7, depth=13, n_pade=2),              # the first with diagonals
    lambda: W.spin_boson_tt(rank=5, depth=40, n_pade=3),
    lambda: W.spin_boson_tt(rank=9, depth=14, n_pade=4, tree="btt"),  # two open legs, shared pairs
    lambda: driven(14),                                               # operators rewritten by a drive
    lambda: W.exciton_chain(n_sites=21, rank=3, depth=2, n_pade=1),   # tables of every size
    lambda: W.spin_boson_tt(rank=64, depth=24, n_pade=3),             # QR of 1536 x 64: one copy of Gram and solves
    lambda: W.spin_boson_tt(rank=64, depth=32, n_pade=3),             # QR of 2048 x 64: in global memory
]


@pytest.mark.parametrize("make", STEPS)
def test_step_matches_the_oracle(pkg, make):
    w = make()
    g, o = pair(pkg, w)
    g.ttn_step(w.dt, pkg.TTN_PS1, 1)
    o.step(w.dt, "ps1")
    assert np.max(np.abs(g.ttn_rdm() - o.rdm())) <= 1e-11
    for u in range(g.n_nodes):
        assert np.max(np.abs(g.ttn_get_node(u) - o.tensors[u])) <= 1e-11, u
    g.close()


def test_job_tables_beyond_the_parameter_sizes(pkg):
    w = STEPS[5]()
    g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0)
    r = g.ttn_tuning_get()
    assert r[r[:, 0] == 0][:, 6].max() > 40  # outputs of one list
    g.close()


@pytest.mark.parametrize("make", [
    lambda: W.exciton_chain(n_sites=45, rank=2, depth=2, n_pade=2),       # up to 64 nodes on a level: two launches
    lambda: W.spin_boson_tt(rank=2, depth=2, n_pade=40),                  # one node on each of 41 levels
    lambda: W.spin_boson_tt(rank=2, depth=2, n_pade=0),                   # the root alone
])
def test_density_matrix_of_wide_and_deep_trees(pkg, make):
    g, o = pair(pkg, make())
    ref = o.rdm()
    assert np.max(np.abs(g.ttn_rdm() - ref)) <= 1e-11 * np.max(np.abs(ref))
    g.close()


@pytest.mark.parametrize("rank,depth,K,tree", [
    (1, 3, 3, "tt"),     # bonds of one
    (9, 14, 5, "btt"),   # operators of three diagonals in the node lists
    (64, 9, 4, "tt"),    # the widest inverse in shared memory
    (66, 9, 4, "tt"),    # in global memory
])
def test_direct_integration_matches_the_oracle(pkg, rank, depth, K, tree):
    w = W.spin_boson_tt(rank=rank, depth=depth, n_pade=K - 1, tree=tree)
    g, o = pair(pkg, w, {"ode_rtol": 1e-7, "ode_atol": 1e-9, "vmf_atol": 1e-3})
    g.ttn_step(0.002, pkg.TTN_VMF, 1)
    o.step(0.002, "vmf")
    assert np.max(np.abs(g.ttn_rdm() - o.rdm())) <= 1e-10
    for u in range(g.n_nodes):
        assert np.max(np.abs(g.ttn_get_node(u) - o.tensors[u])) <= 1e-10, u
    g.close()


@pytest.mark.parametrize("make", STEPS[1:5:3])
def test_overlapped_launches_on_the_default_stream(pkg, make):
    """Launch by launch on the legacy default stream, as a graph on a stream of its
    own, and launch by launch there: the same bits (every kernel waits for the one before)."""
    import torch
    w = make()
    out = []
    for stream, prof in ((torch.cuda.default_stream(), 0), (None, 0), (None, 1)):
        g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, drives=w.drives,
                           stream=stream)
        g.ttn_profile(prof)
        g.ttn_step(w.dt, pkg.TTN_PS1, 5)
        out.append([g.ttn_rdm()] + [g.ttn_get_node(u) for u in range(g.n_nodes)])
        g.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
