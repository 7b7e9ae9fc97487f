"""Arc walks are cut into tasks whose length follows the graph's arcs (128 to
2 048 per warp): one bad arc anywhere -- the first, the last, either side of a
task's edge -- is still found by the checks at load, and the in-arc CSR and the
level sums that follow from it are the oracle's, at sizes around the edges."""
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


def _chunk(arcs):
    return min(2048, max(128, -(-(arcs // 8192) // 32) * 32))


def _refused(t, ctx, n, off, cols, directed):
    with pytest.raises(t.TkcError) as err:
        t.tkc_free_graph(t.tkc_load_csr(ctx, n, off, cols, directed))
    assert err.value.code == t.TKC_EGRAPH


# paths: 2 (n - 1) arcs, so 126, 128, 130, ... arcs around the tasks of 128;
# the last two are cut into tasks of 160 and 2 048
@pytest.mark.parametrize("n", [2, 17, 64, 65, 66, 2049, 600_000, 9_000_000])
def test_one_bad_arc_is_found(gpu_lib, ctx, n):
    t = gpu_lib
    g = gg.path(n)
    arcs, c = g.arcs, _chunk(g.arcs)
    t.tkc_free_graph(t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, False))
    for e in sorted({0, arcs - 1, min(c, arcs) - 1, min(c, arcs - 1), (arcs // c) * c - (arcs % c == 0)}):
        cols = g.cols.copy()
        cols[e] = n  # out of range
        _refused(t, ctx, n, g.offsets, cols, False)
        src = int(np.searchsorted(g.offsets, e, side="right")) - 1
        cols[e] = src  # a self-loop
        _refused(t, ctx, n, g.offsets, cols, True)
        if n > 4:  # an arc moved to another target: its reverse is missing
            cols[e] = g.cols[e]
            row = cols[g.offsets[src]:g.offsets[src + 1]]
            row[:] = np.sort(np.concatenate([np.setdiff1d(row, [g.cols[e]]),
                                             [src + 3 if src + 3 < n else src - 3]])).astype(np.uint32)
            _refused(t, ctx, n, g.offsets, cols, False)


@pytest.mark.parametrize("n", [17, 32, 33, 3000])
def test_reach_bounds_and_sums(gpu_lib, ctx, n):
    t = gpu_lib
    g = gg.erdos_renyi(n, 4 * n, n)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, True)
    try:
        a, o = t.tkc_reach_bounds(h, n)
        wa, wo = oracle.alpha_omega(g)
        assert np.array_equal(a, wa) and np.array_equal(o, wo)
        S, r = t.tkc_distance_sums(h, np.arange(n))
        wS, wr = oracle.bfs_sums(g, np.arange(n, dtype=np.uint32))
        assert np.array_equal(S, wS) and np.array_equal(r, wr)
    finally:
        t.tkc_free_graph(h)
