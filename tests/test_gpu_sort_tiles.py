"""The radix sort where its tiles change: tiles of 1 024 up to 131 072 pairs and
of 4 096 up to 524 288, both with the digit counts added up by every block, and
tiles of 4 096 behind a scan beyond.  One to three passes, an uneven last tile."""
import numpy as np
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = gpu_lib.tkc_create(gpu_lib.Options())
    yield c
    gpu_lib.tkc_destroy(c)


@pytest.mark.parametrize("max_degree", [200, 60000, 100000])
@pytest.mark.parametrize("n", [8193, 9217, 131071, 131072, 131073, 135169, 524287, 524288, 524289, 528385])
def test_degree_order_is_stable_by_id(gpu_lib, ctx, n, max_degree):
    t = gpu_lib
    rng = np.random.default_rng(n + max_degree)
    hub = min(max_degree, n - 1)
    # one vertex of the largest degree, the others 0 to 4 or (some) hundreds
    deg = rng.integers(0, 5, n)
    some = rng.integers(0, n, 300)
    deg[some] = rng.integers(0, min(hub, 400) + 1, 300)
    deg[n // 2] = hub
    src = np.repeat(np.arange(n, dtype=np.int64), deg)
    first = np.zeros(n + 1, np.int64)
    np.cumsum(deg, out=first[1:])
    dst = (src + 1 + np.arange(len(src)) - first[src]) % n
    g = gg.from_arcs(n, src, dst, True)
    assert np.array_equal(g.outdeg(), deg)
    h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
    try:
        assert np.array_equal(t.tkc_source_order(h, n), np.lexsort((np.arange(n), -deg)))
    finally:
        t.tkc_free_graph(h)
