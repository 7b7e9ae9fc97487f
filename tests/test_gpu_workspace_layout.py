"""One context for graphs of different sizes, team counts and batch widths: the
per-team buffers are laid out for each run anew (tests/oracle results whatever
ran before), and a small graph's many teams do not size a large graph's memory."""
import numpy as np
import pytest

import oracle
from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
K = 10


@pytest.fixture(scope="module")
def graphs():
    gs = [gg.rmat(13, 8, seed=4), gg.barabasi_albert(30_001, 3, 5), gg.barabasi_albert(999, 3, 6), gg.rmat(14, 8, seed=9)]
    return [(g, oracle.textbook_topk(g, K, threads=0)) for g in gs]


def _load(t, ctx, g):
    return t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)


@pytest.mark.parametrize("widths", [(0, 0, 0, 0), (512, 64, 128, 256), (64, 512, 1, 128)])
def test_alternating_runs(gpu_lib, graphs, widths):
    t = gpu_lib
    ctx = t.tkc_create()
    try:
        for teams in (0, 1, 37, 0):
            for (g, ref), bits in zip(graphs, widths):
                for order in (t.TKC_ORDER_NB, t.TKC_ORDER_DEG):
                    t.tkc_set_options(ctx, t.Options(order=order, batch_bits=bits, teams=teams))
                    h = _load(t, ctx, g)
                    res = t.tkc_topk_closeness(h, K)
                    S, r = t.tkc_distance_sums(h, np.r_[ref.ids, np.arange(0, 640, dtype=np.uint32)])
                    t.tkc_free_graph(h)
                    assert list(res.ids) == list(ref.ids) and np.array_equal(res.dist_sum, ref.S), (g.n, bits, teams)
                    assert np.array_equal(S[:K], ref.S) and np.array_equal(r[:K], ref.r), (g.n, bits, teams)
    finally:
        t.tkc_destroy(ctx)


def test_many_teams_before_a_large_graph(gpu_lib, graphs):
    """Complete searches of a small graph use a team per batch (64 here); 64 sets
    of rows and lists for 300 000 vertices would take 1.7 GB, the few teams of
    the large graph's search take 0.1."""
    import torch

    t = gpu_lib
    big = gg.barabasi_albert(300_000, 4, 8)

    def held(small_first):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = t.tkc_create(t.Options(order=t.TKC_ORDER_NB))
        try:
            if small_first:
                h = _load(t, ctx, graphs[0][0])
                t.tkc_distance_sums(h, np.arange(0, 4096, dtype=np.uint32))
                assert t.tkc_last_run_stats(ctx)["teams"] >= 32
                t.tkc_free_graph(h)
            h = _load(t, ctx, big)
            res = t.tkc_topk_closeness(h, K)
            t.tkc_free_graph(h)
            return before - torch.cuda.mem_get_info()[0], list(res.ids)
        finally:
            t.tkc_destroy(ctx)

    alone, want = held(False)
    after, got = held(True)
    assert got == want
    assert after < alone + (512 << 20)
