"""Several graphs in one launch beside a program that holds most of the card: the
library's team count follows what is free, and is lowered when an allocation
fails all the same.  Results never depend on it."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
GB = 1 << 30


def _run(t, ctx, gs, k=5):
    hs = t.tkc_load_csr_many(ctx, [(g.n, g.offsets, g.cols, g.directed) for g in gs])
    try:
        res = t.tkc_topk_closeness_multi(ctx, hs, k)
    finally:
        for h in hs:
            t.tkc_free_graph(h)
    return [(list(r.ids), list(r.dist_sum), list(r.reach)) for r in res], t.tkc_last_run_stats(ctx)["teams"]


def test_beside_a_full_card(gpu_lib):
    """3 million vertices: 38 teams of 128-bit rows would take 10 GB; 5 are free."""
    import torch

    t = gpu_lib
    gs = [gg.barabasi_albert(250_000, 3, 10 + i) for i in range(12)]
    ctx = t.tkc_create(t.Options(order=t.TKC_ORDER_NB))
    want, teams = _run(t, ctx, gs)
    t.tkc_destroy(ctx)
    assert teams >= 30
    ctx = t.tkc_create(t.Options(order=t.TKC_ORDER_NB))
    hold = None
    try:
        torch.cuda.synchronize()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - 5 * GB, dtype=torch.uint8, device="cuda")
        got, fewer = _run(t, ctx, gs)
        assert 1 <= fewer < teams and got == want
        assert torch.cuda.mem_get_info()[0] > GB  # it did not take all that was left
        del hold
        hold = None
        torch.cuda.empty_cache()
        got, again = _run(t, ctx, gs)
        assert again == teams and got == want
    finally:
        del hold
        torch.cuda.empty_cache()
        t.tkc_destroy(ctx)


@pytest.mark.parametrize("call", ["multi", "topk"])
def test_fewer_teams_after_a_failed_allocation(gpu_lib, call):
    """The allocations of one call, one by one, find no memory once (counted on the
    host; the retry finds it again): the call either reports it or answers."""
    t = gpu_lib
    fn = t._lib.tkc_internal_fail_allocation_once
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_uint64], ctypes.c_uint64
    gs = [gg.barabasi_albert(40_000, 3, 4), gg.rmat(15, 6, seed=5)]
    refs = [oracle.textbook_topk(g, 5, threads=0) for g in gs]
    answered = set()
    for nth in range(1, 400):
        ctx = t.tkc_create(t.Options(order=t.TKC_ORDER_DEG))
        try:
            hs = t.tkc_load_csr_many(ctx, [(g.n, g.offsets, g.cols, g.directed) for g in gs])
            fn(ctx, nth)
            try:
                res = t.tkc_topk_closeness_multi(ctx, hs, 5) if call == "multi" else [t.tkc_topk_closeness(hs[0], 5)]
                for r, ref in zip(res, refs):
                    assert list(r.ids) == list(ref.ids) and np.array_equal(r.dist_sum, ref.S)
                answered.add(t.tkc_last_run_stats(ctx)["teams"])
            except t.TkcError as e:
                assert e.code == t.TKC_ENOMEM
            left = fn(ctx, 0)
            for h in hs:
                t.tkc_free_graph(h)
        finally:
            t.tkc_destroy(ctx)
        if left:
            break
    assert left and len(answered) == 2  # the full count, and half of it
