"""Rounds that run inside one cooperative launch: trimming, colouring and
Algorithm 6 (directed reach bounds), components (undirected), NB sweeps.
Graphs with many rounds of each, a target of more than 4 096 predecessors, and
sizes either side of the line up to which all sweeps share a launch, against
the oracle."""
import numpy as np
import pytest

import oracle
from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = gpu_lib.tkc_create(gpu_lib.Options())
    yield c
    gpu_lib.tkc_destroy(c)


def _cycle_chain(cycles, length, seed):
    """Directed cycles of one length, each reaching some later ones; ids shuffled."""
    rng = np.random.default_rng(seed)
    n = cycles * length
    src = np.arange(n)
    dst = src - src % length + (src + 1) % length
    a = rng.integers(0, cycles - 1, 2 * cycles)
    b = a + 1 + (rng.random(2 * cycles) * (cycles - 1 - a)).astype(np.int64)
    src = np.concatenate([src, a * length])
    dst = np.concatenate([dst, b * length])
    perm = rng.permutation(n)
    return gg.from_arcs(n, perm[src], perm[dst], True)


def _fan(k):
    """k vertices into a 3-cycle, which reaches k others."""
    src = np.concatenate([np.arange(k), [k, k + 1, k + 2], np.full(k, k)])
    dst = np.concatenate([np.full(k, k), [k + 1, k + 2, k], np.arange(k + 3, 2 * k + 3)])
    return gg.from_arcs(2 * k + 3, src, dst, True)


@pytest.mark.parametrize("make", [
    lambda: gg.path(3000, directed=True), lambda: _cycle_chain(200, 3, 1), lambda: _cycle_chain(40, 50, 2),
    lambda: _fan(5000), lambda: gg.rmat(13, 4, seed=9), lambda: gg.from_arcs(1, [], [], True),
    lambda: gg.disjoint_union(*[gg.cycle(k, True) for k in range(3, 40)]),
])
def test_directed_reach_bounds(gpu_lib, ctx, make):
    t, g = gpu_lib, make()
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, True)
    try:
        a, o = t.tkc_reach_bounds(h, g.n)
        wa, wo = oracle.alpha_omega(g)
        assert np.array_equal(a, wa) and np.array_equal(o, wo)
    finally:
        t.tkc_free_graph(h)


@pytest.mark.parametrize("n", [33, 20000])
def test_components(gpu_lib, ctx, n):
    t = gpu_lib
    rng = np.random.default_rng(n)
    perm = rng.permutation(n)
    cut = np.flatnonzero(rng.random(n - 1) > 0.01)  # a path broken in about n / 100 places, ids shuffled
    g = gg.from_arcs(n, perm[cut], perm[cut + 1], False)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, False)
    try:
        a, o = t.tkc_reach_bounds(h, n)
        piece = np.concatenate([[0], np.cumsum(~np.isin(np.arange(n - 1), cut))])
        size = np.bincount(piece)[piece]
        want = np.empty(n, np.int64)
        want[perm] = size
        assert np.array_equal(a, want) and np.array_equal(o, want)
    finally:
        t.tkc_free_graph(h)


@pytest.mark.parametrize("n", [1, 2, 31, 3001, 1 << 17, (1 << 17) + 1])
@pytest.mark.parametrize("directed", [False, True])
def test_nb_sweeps(gpu_lib, ctx, n, directed):
    t = gpu_lib
    if directed:
        g = gg.erdos_renyi(n, 3 * n, n) if n > 2 else gg.path(n, directed=True)
    else:  # a hub of n / 2 spokes (segmented gather from 2 048 up) and a tail
        half = n // 2
        g = gg.from_arcs(n, np.concatenate([np.zeros(max(half - 1, 0), np.int64), np.arange(half, max(n - 1, half))]),
                         np.concatenate([np.arange(1, max(half, 1)), np.arange(half + 1, max(n, half + 1))]), False)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for levels in (1, 2, 3, 40):
            nb, want = t.tkc_nb_bounds(h, n, levels), oracle.nb_bounds(g, max_levels=levels)
            assert np.array_equal(nb.S, want.S) and np.array_equal(nb.r, want.r), levels
            assert np.array_equal(nb.key, want.key) and nb.levels == want.levels, levels
    finally:
        t.tkc_free_graph(h)
