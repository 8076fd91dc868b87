"""FP64 contractions and projections by the exact digit split, output by output
against extended-precision sums and against the multiply-add chain of the
CUDA-core kernels: gradings of the operands, every number of row blocks, and
non-finite operands; and whole runs against the chain's.

Bound: the split drops less than 2^-56.8 of (row scale x position scale) for each
real product, and outputs whose products sum to less than 2^-12 of those scales
are made by the chain, so a part of an output of n real products is within
n 2^-44.8 sum |a b|; the roundings of the chain and of the sums over terms and
chunks, n 2^-53 sum |a b|, are below the digits of that figure. As a root mean
square over the outputs the error is no larger than the chain's."""
import os
import struct
import subprocess

import numpy as np
import pytest

from paper_2603_17711_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    lib = build.build()
    exe = str(tmp_path_factory.mktemp("harness") / "split_harness")
    subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "-I", build.CSRC, os.path.join(HERE, "split_harness.cu"),
                    lib, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib), "-o", exe], check=True, capture_output=True)
    return exe


def call(exe, project, dims, legs, arrays, shape, chain=0, max_split=1):
    d = tuple(dims) + (1,) * (4 - len(dims))
    data = struct.pack("<8i", project, chain, *d, len(legs), max_split) + np.asarray(legs, "<i4").tobytes()
    data += b"".join(np.ascontiguousarray(a, "<c16").tobytes() for a in arrays)
    r = subprocess.run([exe], input=data, capture_output=True)
    assert r.returncode == 0, r.stderr
    taken, status = struct.unpack_from("<2i", r.stdout)
    assert taken == 1 and status == 0  # the list is one of those that take this path
    return np.frombuffer(r.stdout, "<c16", offset=8).reshape(shape)


def product(M, leg, X):
    """(re, im, sum |a b|) of M x_leg X in extended precision."""
    mr, mi, xr, xi = (np.asarray(v, np.longdouble) for v in (M.real, M.imag, X.real, X.imag))
    f = lambda a, b: np.moveaxis(np.tensordot(a, b, axes=(1, leg)), 0, leg)  # noqa: E731
    return f(mr, xr) - f(mi, xi), f(mr, xi) + f(mi, xr), f(abs(M), abs(X))


def check(split, chain, terms, n):
    re, im, size = (sum(v) for v in zip(*terms))
    assert np.all(np.abs(split.real - re) <= n * 2.0 ** -44.8 * size)
    assert np.all(np.abs(split.imag - im) <= n * 2.0 ** -44.8 * size)
    rms = lambda y: float(np.sqrt(np.mean(((y.real - re) ** 2 + (y.imag - im) ** 2) / size ** 2)))  # noqa: E731
    assert rms(split) <= rms(chain)


def cnormal(rng, shape):
    return rng.normal(size=shape) + 1j * rng.normal(size=shape)


def graded(kind, rng, d, dims, leg):
    """An operator and a tensor of the given grading along the contracted leg."""
    M, X = cnormal(rng, (d, d)), cnormal(rng, dims)
    x = np.arange(d)
    g = 10.0 ** (-12.0 * x / d)  # one to 1e-12
    at = lambda v: v.reshape([d if i == leg else 1 for i in range(len(dims))])  # noqa: E731
    if kind == "product":  # row x position, on both operands
        M, X = M * g[:, None] * g[None, ::-1], X * at(g)
    elif kind == "coupled":  # weak directions coupled to themselves by 1, to the others by 1e-9
        M, X = np.eye(d) + 1e-9 * M, X * at(g)
    elif kind == "diagonal":  # 10^(-0.6 |x - n|): a nearly diagonal isometry
        other = [i for i in range(len(dims)) if i != leg][0]
        n = np.arange(dims[other]).reshape([dims[other] if i == other else 1 for i in range(len(dims))])
        M, X = np.eye(d) + 1e-9 * M, X * 10.0 ** (-0.6 * np.abs(at(x) - n))
    elif kind in ("one", "half"):  # rows that see only x's that are small at positions where others are large
        few = x < (1 if kind == "one" else d // 2)
        M = np.where(x[:, None] % 2 == 0, M * few[None, :], M)
        X = X * np.where(at(few), 1e-12, 1.0)
        X[tuple(0 if i != leg else slice(None) for i in range(len(dims)))] = 1.0
    elif kind == "parts":  # almost real operands
        M, X = M.real + 1e-13j * M.imag, X.real + 1e-11j * X.imag
    return M, X


# 8-row blocks 3 .. 8 of the contracted leg, full and ragged; three and four legs
SHAPES = [((64, 20, 19), 0), ((20, 57, 21), 1), ((21, 20, 49), 2), ((41, 24, 23), 0), ((33, 30, 18), 0),
          ((25, 25, 25), 1), ((17, 33, 33), 0), ((6, 20, 5, 40), 3)]


@pytest.mark.parametrize("dims,leg", SHAPES)
@pytest.mark.parametrize("kind", ["flat", "product", "coupled", "diagonal", "one", "half", "parts"])
def test_every_component_of_a_contraction(harness, dims, leg, kind):
    d = dims[leg]
    rng = np.random.default_rng(d)
    n_terms = -(-int(8e6) // (8 * int(np.prod(dims)) * d))
    ops = [graded(kind, rng, d, dims, leg) for _ in range(n_terms)]
    X = ops[0][1]
    split, chain = (call(harness, 0, dims, [leg] * n_terms, [M for M, _ in ops] + [X], dims, c) for c in (0, 1))
    check(split, chain, [product(M, leg, X) for M, _ in ops], 2 * d * n_terms)


@pytest.mark.parametrize("dims,leg", [((64, 40, 41), 0), ((48, 57, 50), 1), ((45, 47, 33), 2), ((25, 60, 61), 0)])
@pytest.mark.parametrize("kind", ["flat", "product", "diagonal", "one", "half", "parts"])
def test_every_component_of_a_projection(harness, dims, leg, kind):
    d = dims[leg]
    rng = np.random.default_rng(d)
    V = graded(kind, rng, d, dims, leg)[1]
    Wt = graded("flat" if kind in ("one", "half") else kind, rng, d, dims, leg)[1]
    split, chain = (call(harness, 1, dims, [leg], [V, Wt], (d, d), c) for c in (0, 1))
    flat = lambda a: np.moveaxis(a, leg, 0).reshape(d, -1)  # noqa: E731
    check(split, chain, [product(flat(V).conj(), 0, flat(Wt).T)], 2 * int(np.prod(dims)) // d)


@pytest.mark.parametrize("kind", ["flat", "diagonal", "half"])
def test_terms_cut_over_several_planes(harness, kind):
    """A tile on more than one CTA (max_split above 1) and terms on every leg."""
    dims, rng = (40, 41, 39), np.random.default_rng(4)
    legs = [0, 1, 2] * 5
    X = graded(kind, rng, 40, dims, 0)[1]
    ops = [graded(kind, rng, dims[leg], (dims[leg], 2), 0)[0] for leg in legs]
    split, chain = (call(harness, 0, dims, legs[:12], ops[:12] + [X], dims, c, 16) for c in (0, 1))
    check(split, chain, [product(M, leg, X) for M, leg in zip(ops[:12], legs)], 2 * 40 * 12)


def test_powers_of_two_and_zeros(harness):
    dims, rng = (33, 32, 31), np.random.default_rng(5)
    M, X = graded("diagonal", rng, 33, dims, 0)
    X[:, 5] = 0.0
    y = call(harness, 0, dims, [0], [M, X], dims)
    z = call(harness, 0, dims, [0], [M * 2.0 ** -300, X * 2.0 ** 340], dims)
    assert np.array_equal(z, y * 2.0 ** 40)
    assert not y[:, 5].any() and y[:, 4].all()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, complex(0.0, np.inf)])
def test_what_is_not_finite_spreads(harness, bad):
    """A non-finite operand makes the outputs that it enters non-finite, and leaves the others as they are."""
    dims, rng = (41, 29, 30), np.random.default_rng(6)
    M, X = cnormal(rng, (41, 41)), cnormal(rng, dims)
    M[9, 2] = X[7, 3, 11] = 0.0
    good = call(harness, 0, dims, [0], [M, X], dims)
    X[7, 3, 11] = bad
    y = call(harness, 0, dims, [0], [M, X], dims)
    hit = np.zeros(dims, bool)
    hit[:, 3, 11] = True
    assert np.array_equal(~np.isfinite(y), hit)
    assert np.array_equal(y[~hit], good[~hit])
    X[7, 3, 11] = 0.0
    M[9, 2] = bad
    y = call(harness, 0, dims, [0], [M, X], dims)
    hit = np.broadcast_to((np.arange(41) == 9)[:, None, None], dims)
    assert np.array_equal(~np.isfinite(y), hit)
    assert np.array_equal(y[~hit], good[~hit])


@pytest.mark.parametrize("args,steps", [(dict(n_sites=3, rank=28, depth=8), 10), (dict(n_sites=4, rank=32, depth=8), 20)])
def test_a_run_keeps_its_weak_directions(args, steps):
    """From the product state on the tensor cores (max_split 1: lists from 8 MFLOP) and
    twice on the CUDA cores (the lists of these sizes stay below 100 MFLOP) in two
    orders of the sums. What the order changes is rounding in the weakly occupied
    directions, 2e-9 and 6e-14 on the nodes; the split may not change more than a
    hundred times that (without its care for weak outputs: 1e-5 and 5e-6)."""
    import workloads as W
    import paper_2603_17711_gb300 as pkg
    w = W.exciton_chain(**args)
    rho, nodes = [], []
    for max_split in (16, 4, 1):
        g = pkg.from_model(w.H, w.baths, w.depth, w.parent, w.leg_node, w.ranks, rho0=w.rho0, params=dict(max_split=max_split))
        g.ttn_step(w.dt, pkg.TTN_PS1, steps)
        rho.append(g.ttn_rdm())
        nodes.append(np.concatenate([g.ttn_get_node(u).reshape(-1) for u in range(g.n_nodes)]))
        g.close()
    noise = np.max(np.abs(nodes[0] - nodes[1]))
    assert np.max(np.abs(nodes[0] - nodes[2])) <= 100 * noise
    assert np.max(np.abs(rho[0] - rho[2])) <= 1e-13
