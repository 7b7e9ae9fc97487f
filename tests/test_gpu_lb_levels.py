"""Level bounds of searches deeper than one step of 32 levels, and rounds of more
than one stage of 512 slots: one source a round with the oracle's counters
(every bound is then pinned by the order it leaves), and wide rounds against the
textbook, twice on one context (the level sizes and rows are left clean)."""
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


GRAPHS = [lambda: gg.path(32), lambda: gg.path(33), lambda: gg.path(34), lambda: gg.cycle(131),
          lambda: gg.grid(3, 64, seed=2, drop=0.05), lambda: gg.grid(4, 50, directed=True, seed=3, drop=0.1),
          lambda: gg.cycle(70, True), lambda: gg.path(100, directed=True),
          lambda: gg.disjoint_union(gg.path(65), gg.cycle(64), gg.star(9))]


def _expect(got, ref, g):
    assert list(got.ids) == list(ref.ids), g.name
    assert np.array_equal(got.dist_sum, ref.S) and np.array_equal(got.reach, ref.r), g.name
    assert got.n_tied_at_kth == ref.n_tied, g.name


@pytest.mark.parametrize("nb", [False, True])
@pytest.mark.parametrize("gi", range(len(GRAPHS)))
def test_deep_searches(gpu_lib, ctx, gi, nb):
    t = gpu_lib
    g = GRAPHS[gi]()
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for k in (1, 10):
            if nb:
                b = oracle.nb_bounds(g)
                order = oracle.nb_order(g, b.key).tolist() + np.nonzero(g.outdeg() == 0)[0].tolist()
                c = oracle.bfsbound(g, k, order, b).counters
            else:
                c = oracle.bfsbound(g, k).counters
            ref = oracle.textbook_topk(g, k)
            for bits, teams in ((1, 0), (64, 0), (0, 0), (64, 9), (512, 2)):
                t.tkc_set_options(ctx, t.Options(order=t.TKC_ORDER_NB if nb else t.TKC_ORDER_DEG, batch_bits=bits, teams=teams))
                for _ in range(2):
                    got = t.tkc_topk_closeness_bound(h, k)
                    _expect(got, ref, g)
                    if bits == 1:
                        assert (got.bfs_started, got.edges_visited) == (c.bfs_started, c.edges_visited), (g.name, k)
    finally:
        t.tkc_free_graph(h)
        t.tkc_set_options(ctx, t.Options())


def test_rounds_of_more_than_one_stage(gpu_lib, ctx):
    t = gpu_lib
    g = gg.grid(40, 45, seed=8, drop=0.1)
    ref = oracle.textbook_topk(g, 10, threads=0)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for bits, teams in ((64, 9), (128, 5), (256, 4), (512, 2)):
            t.tkc_set_options(ctx, t.Options(order=t.TKC_ORDER_NB, batch_bits=bits, teams=teams))
            _expect(t.tkc_topk_closeness_bound(h, 10), ref, g)
    finally:
        t.tkc_free_graph(h)
        t.tkc_set_options(ctx, t.Options())
