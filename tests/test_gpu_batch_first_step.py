"""The first batched step on new handles: the members' steps are captured, and one
executable graph is made of them, none of each."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def handles(pkg, n):
    out = []
    for i in range(n):
        w = W.spin_boson_tt(depth=4 + i, rank=4, n_pade=2)
        out.append((w, pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0)))
    return out


def test_one_executable_graph_for_the_batch():
    import torch
    from torch.profiler import ProfilerActivity, profile
    import paper_2603_17711_gb300 as pkg
    hs = handles(pkg, 3)
    dt = hs[0][0].dt
    with profile(activities=[ProfilerActivity.CUDA]):  # the first one sets the profiler up
        hs[0][1].ttn_rdm()
    with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
        pkg.ttn_batch_step([h for _, h in hs], dt, pkg.TTN_PS1, 1)
        torch.cuda.synchronize()
    calls = {e.key: e.count for e in prof.key_averages() if "Graph" in e.key}
    assert sum(v for k, v in calls.items() if "Instantiate" in k) == 1, calls
    # a member on its own, and the batch after one of them was captured anew
    hs[1][1].ttn_step(dt, pkg.TTN_PS1, 1)
    hs[1][1].ttn_set_params(kappa=5.0)
    pkg.ttn_batch_step([h for _, h in hs], dt, pkg.TTN_PS1, 2)
    for i, (w, h) in enumerate(handles(pkg, 3)):
        h.ttn_step(dt, pkg.TTN_PS1, 1)
        if i == 1:
            h.ttn_step(dt, pkg.TTN_PS1, 1)
            h.ttn_set_params(kappa=5.0)
        h.ttn_step(dt, pkg.TTN_PS1, 2)
        assert np.array_equal(h.ttn_rdm(), hs[i][1].ttn_rdm())
        h.close()
        hs[i][1].close()
