"""The host's launch counters against the kernels that ran."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2603_17711_gb300 as p
    p.library()
    return p


def make(pkg, w, **kw):
    return pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, **kw)


@pytest.mark.parametrize("rank,precision", [(20, "fp64"), (40, "fp64"), (64, "fp64"), (64, "mixed")])
def test_launches_are_those_of_the_step(pkg, rank, precision):
    """Lists of several launches (the digit split's planes and their sum, the
    FP32 tensor-core lists, the blocked QR) count each of them: as many as the
    profiler sees kernels."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    w = W.exciton_chain(n_sites=2, rank=rank, depth=8)
    g = make(pkg, w, precision=pkg.TTN_FP64 if precision == "fp64" else pkg.TTN_MIXED_FP32)
    g.ttn_step(w.dt, pkg.TTN_PS1, 1)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]):  # the first one sets the profiler up
        g.ttn_step(w.dt, pkg.TTN_PS1, 1)
        torch.cuda.synchronize()
    g.ttn_stats_reset()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        g.ttn_step(w.dt, pkg.TTN_PS1, 1)
        torch.cuda.synchronize()
    seen = {e.key: e.count for e in prof.key_averages() if "ttn::" in e.key}
    assert seen and sum(g.ttn_stats(k)[0] for k in range(4)) == sum(seen.values()), seen
    g.close()
