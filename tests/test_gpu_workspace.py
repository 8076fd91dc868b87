"""A workspace that ends before the digit split's planes (the size asked for by
handles without it) is accepted, gives the same steps, and is not written past."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = [  # model, scheme, bytes without the planes
    (lambda: W.driven_structured_tls(n_steps=1, n_pade=1, depth=10, cap=16), "ps2", 16123136),
    (lambda: W.exciton_chain(n_sites=2, rank=40, depth=8), "ps1", 34557440),  # lists that use the planes
    (lambda: W.spin_boson_tt(rank=10, depth=10, n_pade=3), "ps1", 20067584),
    (lambda: W.exciton_chain(n_sites=4, rank=3, depth=3, n_pade=0), "ps1", 3896832),
    (lambda: W.spin_boson_tt(rank=4, depth=3, n_pade=0), "ps1", 1778688),
    (lambda: W.exciton_chain(rank=20), "ps1", 902682880),
]


def handle(pkg, w):
    params = dict(max_rank=16, ps2_atol=1e-6) if w.drives else None
    g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, drives=w.drives, params=params)
    return g


@pytest.mark.parametrize("make,scheme,size", CASES)
def test_a_workspace_without_the_planes(make, scheme, size):
    import torch
    import paper_2603_17711_gb300 as pkg
    w = make()
    scheme = pkg.TTN_PS2 if scheme == "ps2" else pkg.TTN_PS1
    full, small = handle(pkg, w), handle(pkg, w)
    assert small.ttn_workspace_size() <= full.ttn_workspace_size()
    guard = 4096
    buf = torch.full((size + guard + 256,), 0x5a, dtype=torch.uint8, device="cuda")
    base = (buf.data_ptr() + 255) // 256 * 256
    off = base - buf.data_ptr()
    torch.cuda.synchronize()
    assert small.lib.ttn_set_workspace(small.h, C.c_void_p(base), size) == 0
    small.ttn_set_rdo0(w.rho0)
    for g in (full, small):
        g.ttn_step(w.dt, scheme, 2)
    assert np.max(np.abs(full.ttn_rdm() - small.ttn_rdm())) <= 1e-12
    assert list(full.ttn_get_ranks()) == list(small.ttn_get_ranks())
    torch.cuda.synchronize()
    assert bool((buf[off + size:off + size + guard] == 0x5a).all())
    assert small.lib.ttn_set_workspace(small.h, C.c_void_p(base), size // 2) != 0  # too small stays refused
    full.close()
    small.close()
