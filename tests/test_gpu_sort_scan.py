"""The radix sort and the scans behind every source order, at the sizes where
their variants meet: one block up to 8 192 elements, tiles of 4 096 beyond;
scans of one block (up to 16 384), of two launches (up to 2^22) and of three."""
import numpy as np
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = gpu_lib.tkc_create(gpu_lib.Options())
    yield c
    gpu_lib.tkc_destroy(c)


def _star_forest(n, seed):
    """Undirected, degrees from 0 to thousands, every degree shared by many vertices."""
    rng = np.random.default_rng(seed)
    hubs = np.minimum((rng.pareto(1.0, n) * 3).astype(np.int64), n - 1)
    return gg.from_arcs(n, np.arange(n), hubs % n, False)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 4095, 4096, 4097, 8191, 8192, 8193, 12289, 16383, 16384, 70001,
                               (1 << 22) - 1, (1 << 22) + 5])
def test_degree_order_is_stable_by_id(gpu_lib, ctx, n):
    t = gpu_lib
    g = _star_forest(n, n)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        want = np.lexsort((np.arange(n), -g.outdeg()))
        assert np.array_equal(t.tkc_source_order(h, n), want)
    finally:
        t.tkc_free_graph(h)


@pytest.mark.parametrize("n", [50, 8192, 8193, 40000])
def test_nb_orders_follow_their_keys(gpu_lib, ctx, n):
    t = gpu_lib
    g = gg.erdos_renyi(n, 5 * n, n)
    src = np.flatnonzero(g.outdeg() > 0)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for levels in (1, 0, 2):  # the orders follow the level cap they are asked for
            hub, horder = t.tkc_nb_harmonic_bounds(h, n, levels)
            nb = t.tkc_nb_bounds(h, n, levels)
            assert np.array_equal(nb.order, src[np.lexsort((src, nb.key[src]))])
            assert np.array_equal(horder, src[np.lexsort((src, -hub[src]))])
    finally:
        t.tkc_free_graph(h)
