"""Which FP64 job lists go to the tensor cores, and that the launcher's host part
serves every list it is offered -- on the plans of real models, without a GPU."""
import os
import subprocess

import numpy as np
import pytest

import workloads as W
from paper_2603_17711_gb300 import build, heom

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    return compile_harness(tmp_path_factory.mktemp("harness"))


def compile_harness(out_dir):
    """The planner and the launcher with the harness, an integer division by zero made fatal on every host."""
    exe = os.path.join(str(out_dir), "lists_harness")
    src = [os.path.join(HERE, "lists_harness.cu")] + [os.path.join(build.CSRC, f) for f in ("plan.cpp", "xs_apply.cu")]
    subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "-I", build.CSRC, "-Xcompiler",
                    "-fsanitize=integer-divide-by-zero,-fno-sanitize-recover=integer-divide-by-zero", *src, "-lubsan", "-o", exe],
                   check=True, capture_output=True)
    return exe


def lists(exe, w, max_split=16):
    """Rows (applicable, launched, outputs, terms, d0, d1, d2, d3) of the model's lists."""
    a = heom.heom_sop(w.H, w.baths, w.depth, w.drives)
    nums = []
    for x in (len(w.parent), w.parent, len(w.leg_node), w.leg_node, w.leg_dims, w.ranks, len(a["op_leg"]), a["op_leg"],
              len(a["op_data"]), a["op_offset"], a["op_data"], len(a["term_offsets"]) - 1, a["term_offsets"],
              len(a["term_ops"]), a["term_ops"], a["coef"], a["coef_drive"], max_split):
        nums += [repr(float(v)) if isinstance(v, (float, np.floating)) else str(int(v)) for v in np.ravel(x)]
    r = subprocess.run([exe, "lists"], input=" ".join(nums), capture_output=True, text=True,
                       env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert r.returncode == 0, (r.returncode, r.stderr)
    return np.array([[int(v) for v in line.split()] for line in r.stdout.splitlines()])


@pytest.mark.parametrize("make", [
    lambda: W.spin_boson_tt(rank=72, depth=8, n_pade=7, tree="btt"),  # nodes 72 x 64 x 64, terms on legs 1 and 2
    lambda: W.exciton_chain(n_sites=3, rank=80, depth=9),
    lambda: W.exciton_chain(n_sites=7, rank=64),
])
def test_a_leg_above_the_limit_that_carries_no_term(harness, make):
    """Legs without a term do not limit the list, and their size divides nothing."""
    r = lists(harness, make())
    assert r[:, 0].any() and np.array_equal(r[:, 0], r[:, 1])


def test_lists_too_long_for_a_launch_are_not_claimed(harness):
    """More than 96 outputs: the list stays with the CUDA-core kernel from the
    start, so the autotuner still finds its tile shape."""
    r = lists(harness, W.exciton_chain(n_sites=60, rank=24, depth=4, n_pade=0))
    assert r[:, 2].max() > 96 and r[:, 0].any()
    assert np.array_equal(r[:, 0], r[:, 1])


def workspace_bytes(w, precision):
    import ctypes as C

    from paper_2603_17711_gb300 import _lib
    build.build()
    lib = _lib.load()
    par, ln = _lib.as_i32(w.parent), _lib.as_i32(w.leg_node)
    tree = _lib.ttn_tree(len(par), _lib.ptr(par, C.c_int32), len(ln), _lib.ptr(ln, C.c_int32))
    h, n = C.c_void_p(), C.c_size_t()
    assert lib.ttn_create(C.byref(tree), _lib.ptr(_lib.as_i32(w.leg_dims), C.c_int32),
                          _lib.ptr(_lib.as_i32(w.ranks), C.c_int32), precision, C.byref(h)) == 0
    a = heom.heom_sop(w.H, w.baths, w.depth)
    assert lib.sop_load(h, len(a["op_leg"]), _lib.ptr(a["op_leg"], C.c_int32), _lib.ptr(a["op_offset"], C.c_int64),
                        _lib.ptr(a["op_data"], C.c_double), len(a["term_offsets"]) - 1,
                        _lib.ptr(a["term_offsets"], C.c_int32), _lib.ptr(a["term_ops"], C.c_int32),
                        _lib.ptr(a["coef"], C.c_double), _lib.ptr(a["coef_drive"], C.c_int32)) == 0
    assert lib.ttn_workspace_size(h, C.byref(n)) == 0
    lib.ttn_destroy(h)
    return n.value


@pytest.mark.parametrize("rank,precision,before", [
    (20, 0, 902682880), (20, 1, 1223671808), (64, 0, 13959593728), (64, 1, 19299940096)])
def test_workspace_without_room_for_planes(rank, precision, before):
    """The mixed form has no digit split and the FP64 form keeps its planes in the
    two-site split's matrices: `before`, the bytes without either, plus the split's
    column counters and pivot candidates (below 32 KiB)."""
    assert workspace_bytes(W.exciton_chain(rank=rank), precision) - before <= 32 << 10


def test_the_two_site_split_has_no_room_of_its_own_either():
    """Its column counters and pivot candidates lie in buffers that are written after them."""
    for rank, precision, before in [(20, 0, 902682880), (20, 1, 1223671808), (64, 0, 13959593728), (64, 1, 19299940096)]:
        assert workspace_bytes(W.exciton_chain(rank=rank), precision) <= before
