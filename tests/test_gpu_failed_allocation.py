"""A device allocation that fails makes its call return TKC_ENOMEM and leaves
the context as good as new: every allocation of a call is made to fail in turn
(counted on the host, nothing is exhausted), and the calls that follow on the
same context, on smaller and on larger graphs, equal the oracle."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
K = 10


@pytest.fixture(scope="module")
def graphs():
    small, large = gg.barabasi_albert(300, 3, 5), gg.rmat(12, 8, seed=7)
    return [(g, oracle.textbook_topk(g, K, threads=0)) for g in (small, large)]


def _arm(t, ctx, nth):
    fn = t._lib.tkc_internal_fail_allocation
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_uint64], ctypes.c_uint64
    return fn(ctx, nth)


def _load(t, ctx, g):
    return t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)


def _is_right(res, ref):
    return list(res.ids) == list(ref.ids) and np.array_equal(res.dist_sum, ref.S) and np.array_equal(res.reach, ref.r)


def _calls(t):
    def shard(h, ctx, gs):
        t.tkc_topk_closeness_shard(h, K, 0, 2)

    def multi(h, ctx, gs):
        hs = t.tkc_load_csr_many(ctx, [(g.n, g.offsets, g.cols, g.directed) for g, _ in gs])
        try:
            t.tkc_topk_closeness_multi(ctx, hs, K)
        finally:
            for x in hs:
                t.tkc_free_graph(x)

    return {"topk": lambda h, ctx, gs: t.tkc_topk_closeness(h, K), "bound": lambda h, ctx, gs: t.tkc_topk_closeness_bound(h, K),
            "harmonic": lambda h, ctx, gs: t.tkc_topk_harmonic(h, K), "shard": shard, "multi": multi,
            "sums": lambda h, ctx, gs: t.tkc_distance_sums(h, np.arange(0, 4000, 3, dtype=np.uint32))}


# wide: batches of 512 for the failing call, whose rows are wider than the next calls'
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("order", ["deg", "nb"])
@pytest.mark.parametrize("call", ["topk", "harmonic", "bound", "shard", "multi", "sums"])
def test_context_survives_every_failure(gpu_lib, graphs, call, order, wide):
    t = gpu_lib
    opts = dict(order=t.TKC_ORDER_NB if order == "nb" else t.TKC_ORDER_DEG)
    run = _calls(t)[call]
    for nth in range(1, 400):
        ctx = t.tkc_create(t.Options(**opts))
        try:
            if nth % 2:  # a workspace from a smaller graph is there, or none
                h = _load(t, ctx, graphs[0][0])
                t.tkc_topk_closeness(h, K)
                t.tkc_free_graph(h)
            t.tkc_set_options(ctx, t.Options(batch_bits=512 if wide else 0, **opts))
            h = _load(t, ctx, graphs[1][0])
            _arm(t, ctx, nth)
            try:
                run(h, ctx, graphs)
                failed = False
            except t.TkcError as e:
                assert e.code == t.TKC_ENOMEM
                failed = True
            reached = _arm(t, ctx, 0) == 0
            assert failed == reached
            t.tkc_free_graph(h)
            t.tkc_set_options(ctx, t.Options(**opts))
            for g, ref in graphs:
                h = _load(t, ctx, g)
                assert _is_right(t.tkc_topk_closeness(h, K), ref), (nth, g.n)
                t.tkc_free_graph(h)
        finally:
            t.tkc_destroy(ctx)
        if not reached:
            break
    assert nth > 10 and not reached
