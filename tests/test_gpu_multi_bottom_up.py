"""Several graphs in one launch: batches of one graph's searches run bottom-up
over that graph's part of the sweep list.  Graphs whose first and last
vertices share frontier-bitmap words with their neighbours (sizes that are not
multiples of 32), with long in-rows, without arcs, with fewer sources than a
batch, at every batch width and several team counts, against the textbook."""
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


def _graphs():
    in_star = gg.from_arcs(333, np.arange(1, 333), np.zeros(332, np.int64), True)  # one row of 332 in-arcs
    return [gg.erdos_renyi(1501, 12008, 1), gg.barabasi_albert(777, 4, 2), gg.path(1), gg.erdos_renyi(31, 120, 3),
            in_star, gg.complete(40), gg.rmat(10, 16, seed=4), gg.erdos_renyi(2049, 16392, 5), gg.path(0),
            gg.barabasi_albert(1023, 3, 6), gg.cycle(97, True)]


_want = {}


def _ref(i, g, k, harmonic):
    key = (i, k, harmonic)
    if key not in _want:
        _want[key] = oracle.textbook_harmonic_topk(g, k) if harmonic else oracle.textbook_topk(g, k)
    return _want[key]


@pytest.mark.parametrize("bits", [0, 64, 128, 256, 512])
@pytest.mark.parametrize("order,teams", [("NB", 0), ("NB", 3), ("DEG", 0), ("DEG", 1)])
def test_every_graph_matches_the_textbook(gpu_lib, ctx, bits, order, teams):
    t = gpu_lib
    gs = _graphs()
    t.tkc_set_options(ctx, t.Options(order=getattr(t, "TKC_ORDER_" + order), batch_bits=bits, teams=teams))
    hs = t.tkc_load_csr_many(ctx, [(g.n, g.offsets, g.cols, g.directed) for g in gs])
    try:
        for k in (1, 10):
            for i, (g, got) in enumerate(zip(gs, t.tkc_topk_closeness_multi(ctx, hs, k))):
                ref = _ref(i, g, k, False)
                assert list(got.ids) == list(ref.ids), (i, k)
                assert np.array_equal(got.dist_sum, ref.S) and np.array_equal(got.reach, ref.r), (i, k)
                assert got.n_tied_at_kth == ref.n_tied, (i, k)
        assert t.tkc_last_run_stats(ctx)["bu_levels"] > 0
        for i, (g, got) in enumerate(zip(gs, t.tkc_topk_harmonic_multi(ctx, hs, 10))):
            ref = _ref(i, g, 10, True)
            assert list(got.ids) == list(ref.ids) and got.n_tied_at_kth == ref.n_tied, i
    finally:
        for h in hs:
            t.tkc_free_graph(h)
