"""The tuner compares its configurations on one labelling of the graph: where a
search of this size may build the labelled copy, it is there before the first is
timed, whether or not a configuration leaves enough batches to build it.  Arcs
scanned by a one-team search tell which labelling it walked."""
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def test_tuned_graph_has_its_copy(gpu_lib):
    t = gpu_lib
    g = gg.rmat(20, 8)
    ctx = t.tkc_create()

    def scanned(relabel, tune=False):
        opts = dict(order=t.TKC_ORDER_DEG, batch_bits=64, teams=1)
        t.tkc_set_options(ctx, t.Options(relabel=relabel, **opts))
        h = t.tkc_load_csr(ctx, g.n, g.offsets, g.cols, g.directed)
        try:
            if tune:
                t.tkc_autotune(h, 10)
            return t.tkc_topk_closeness(h, 10).edges_scanned
        finally:
            t.tkc_free_graph(h)

    try:
        plain, copy = scanned(2), scanned(1)
        # (an in-row holds its arcs in the order the build reached them: counts of one labelling differ a little)
        assert abs(plain - copy) > 0.05 * plain
        assert abs(scanned(0) - plain) < 0.01 * plain
        assert abs(scanned(0, tune=True) - copy) < 0.01 * copy
    finally:
        t.tkc_destroy(ctx)
