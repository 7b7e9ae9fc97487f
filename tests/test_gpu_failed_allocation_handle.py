"""A graph handle stays usable after a call on it failed for lack of device
memory: what the call had begun (in-arc CSR, features, labelled copy, NB bounds,
a given order) is made again, whole.  Every allocation of the call fails in
turn, counted on the host; the same call on the same handle then gives what a
fresh handle gives."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
K = 10


@pytest.fixture(scope="module", params=["directed", "undirected"])
def graph(request):
    g = gg.rmat(11, 8, seed=3) if request.param == "directed" else gg.barabasi_albert(1500, 3, 2)
    return g, oracle.textbook_topk(g, K, threads=0)


def _arm(t, ctx, nth):
    fn = t._lib.tkc_internal_fail_allocation
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_uint64], ctypes.c_uint64
    return fn(ctx, nth)


def _load(t, ctx, g):
    return t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)


def _top(t, g):
    return lambda h: [np.asarray(a) for r in [t.tkc_topk_closeness(h, K)] for a in (r.ids, r.dist_sum, r.reach)]


def _given(t, g):
    order = np.random.default_rng(1).permutation(g.n).astype(np.uint32)

    def run(h):
        t.tkc_set_source_order(h, order)
        return _top(t, g)(h)

    return run


def _bounds(t, g):
    def run(h):
        b = t.tkc_nb_bounds(h, g.n)
        return [np.asarray(x) for x in (b.S, b.r, b.key, b.order)]

    return run


CASES = {
    "top": (dict(), _top),
    "top_nb": (dict(order="TKC_ORDER_NB"), _top),
    "labelled": (dict(relabel=1), _top),
    "learned": (dict(order="TKC_ORDER_LEARNED"), _top),
    "learned_nb": (dict(order="TKC_ORDER_LEARNED_NB", seed_factor=2), _top),
    "given": (dict(order="TKC_ORDER_GIVEN"), _given),
    "reach": (dict(), lambda t, g: lambda h: list(t.tkc_reach_bounds(h, g.n))),
    "nb": (dict(), _bounds),
    "features": (dict(), lambda t, g: lambda h: [t.tkc_vertex_features(h, g.n).cpu().numpy()]),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_handle_survives_every_failure(gpu_lib, graph, case):
    t = gpu_lib
    g, ref = graph
    opts, make = CASES[case]
    opts = {k: getattr(t, v) if isinstance(v, str) else v for k, v in opts.items()}
    run = make(t, g)
    ctx = t.tkc_create(t.Options(**opts))
    try:
        t.tkc_mlp_init(ctx, 3)
        h = _load(t, ctx, g)
        want = run(h)
        t.tkc_free_graph(h)
        if make in (_top, _given):
            assert list(want[0]) == list(ref.ids) and np.array_equal(want[1], ref.S)
        for nth in range(1, 400):
            h = _load(t, ctx, g)
            _arm(t, ctx, nth)
            try:
                run(h)
            except t.TkcError as e:
                assert e.code == t.TKC_ENOMEM
            reached = _arm(t, ctx, 0) == 0
            got = run(h)
            assert len(got) == len(want)
            for a, b in zip(got, want):
                if case == "features":  # standardised by sums that blocks add in any order
                    np.testing.assert_allclose(a, b, rtol=1e-4, atol=1e-5)
                else:
                    assert np.array_equal(a, b), nth
            t.tkc_free_graph(h)
            if not reached:
                break
        assert nth > 2 and not reached
    finally:
        t.tkc_destroy(ctx)


def test_no_order_is_set_by_a_failed_call(gpu_lib, graph):
    t = gpu_lib
    g, _ = graph
    ctx = t.tkc_create(t.Options(order=t.TKC_ORDER_GIVEN))
    try:
        for nth in (1, 2, 3, 4):
            h = _load(t, ctx, g)
            _arm(t, ctx, nth)
            with pytest.raises(t.TkcError) as e:
                t.tkc_set_source_order(h, np.arange(g.n, dtype=np.uint32))
            _arm(t, ctx, 0)
            assert e.value.code == t.TKC_ENOMEM
            with pytest.raises(t.TkcError) as e:
                t.tkc_topk_closeness(h, K)
            assert e.value.code == t.TKC_EINVAL
            t.tkc_free_graph(h)
    finally:
        t.tkc_destroy(ctx)
