"""The filter between the opening and the main launch: sources that the
opening's thresholds abandon (NB stop, level-0 bound, level-1 bound) are
dropped in one pass.  Source counts around its tile edges, lists longer than
one batch (an opening of several batches), uncut prefixes that reach past the
opening, and several graphs in one launch, against the textbook oracle."""
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


def _same(got, ref):
    assert list(got.ids) == list(ref.ids)
    assert np.array_equal(got.dist_sum, ref.S) and np.array_equal(got.reach, ref.r)
    assert got.n_tied_at_kth == ref.n_tied
    assert got.bfs_cut + got.bfs_finished == got.bfs_started


# rest of the order after a 64-source opening: 0, 1, 255, 256, 257 and a ragged larger one
@pytest.mark.parametrize("n", [64, 65, 319, 320, 321, 2999])
@pytest.mark.parametrize("order", ["DEG", "NB"])
@pytest.mark.parametrize("directed", [False, True])
def test_source_counts_around_the_tiles(gpu_lib, ctx, n, order, directed):
    t = gpu_lib
    g = gg.erdos_renyi(n, 12 * n, 7 + n, directed=True) if directed else gg.barabasi_albert(n, 3, 5 + n)
    t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order), batch_bits=64))
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for k in (1, 10, 70):  # 70: the opening is two batches
            _same(t.tkc_topk_closeness(h, k), oracle.textbook_topk(g, k))
        hr, want = t.tkc_topk_harmonic(h, 10), oracle.textbook_harmonic_topk(g, 10)
        assert list(hr.ids) == list(want.ids) and hr.n_tied_at_kth == want.n_tied
    finally:
        t.tkc_free_graph(h)


# skewed in-degrees: the level-2 bound by in-degree class does the pruning;
# harmonic and closeness, one graph in its own ids and in the labelled copy
@pytest.mark.parametrize("scale", [8, 11, 13])
@pytest.mark.parametrize("order", ["DEG", "NB"])
@pytest.mark.parametrize("relabel", [0, 1])
def test_level_2_by_in_degree_class(gpu_lib, ctx, scale, order, relabel):
    t = gpu_lib
    g = gg.rmat(scale, 8, seed=scale)
    t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order), batch_bits=64, relabel=relabel))
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        for k in (1, 10, 100):
            _same(t.tkc_topk_closeness(h, k), oracle.textbook_topk(g, k))
        hr, want = t.tkc_topk_harmonic(h, 10), oracle.textbook_harmonic_topk(g, 10)
        assert list(hr.ids) == list(want.ids) and hr.n_tied_at_kth == want.n_tied
    finally:
        t.tkc_free_graph(h)


# more sources than the pool the opening is picked from (16 384), and a GIVEN
# order that puts the most central vertices last, outside the pool
@pytest.mark.parametrize("n", [16384, 16385, 17001])
def test_order_longer_than_the_pool(gpu_lib, ctx, n):
    t = gpu_lib
    g = gg.barabasi_albert(n, 3, n)
    ref = oracle.textbook_topk(g, 10)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        t.tkc_set_source_order(h, np.argsort(g.outdeg(), kind="stable").astype(np.uint32))
        for order in ("DEG", "NB", "GIVEN"):
            t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order)))
            _same(t.tkc_topk_closeness(h, 10), ref)
    finally:
        t.tkc_free_graph(h)


@pytest.mark.parametrize("seed_factor", [1, 6, 30])  # prefixes of 10, 60 and 300 sources, the opening is 64
@pytest.mark.parametrize("order", ["LEARNED", "LEARNED_NB"])
def test_uncut_prefix_past_the_opening(gpu_lib, ctx, order, seed_factor):
    t = gpu_lib
    g = gg.rmat(11, 16, seed=3)
    t.tkc_mlp_init(ctx, 11)
    t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order), batch_bits=64, seed_factor=seed_factor))
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        got = t.tkc_topk_closeness(h, 10)
        _same(got, oracle.textbook_topk(g, 10))
        assert got.bfs_finished >= min(10 * seed_factor, int((g.outdeg() > 0).sum()))
    finally:
        t.tkc_free_graph(h)


@pytest.mark.parametrize("order", ["DEG", "NB"])
def test_many_graphs(gpu_lib, ctx, order):
    t = gpu_lib
    graphs = [gg.star(3), gg.barabasi_albert(500, 3, 1), gg.erdos_renyi(700, 5000, 2), gg.path(130), gg.cycle(64),
              gg.erdos_renyi(65, 400, 3), gg.barabasi_albert(321, 2, 4)]
    t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order), batch_bits=64))
    hs = t.tkc_load_csr_many(ctx, [(g.n, g.offsets, g.cols, g.directed) for g in graphs])
    try:
        for k in (1, 10):
            for g, got in zip(graphs, t.tkc_topk_closeness_multi(ctx, hs, k)):
                _same(got, oracle.textbook_topk(g, k))
    finally:
        for h in hs:
            t.tkc_free_graph(h)
