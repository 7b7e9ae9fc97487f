"""CSRs on the device whose offsets break the rules while they name arcs: the
check walks those offsets before anything has vouched for them, and reports
them.  (The walk's arithmetic on such offsets is tested on the host.)"""
import numpy as np
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def _bad(n, kind):
    g = gg.path(n, directed=True)
    off, col = g.offsets.astype(np.int64), g.cols.astype(np.int64)
    if kind == "first":
        off[0] = 1
    elif kind == "all":
        off = off + 1
    elif kind == "decreasing":
        off = off[::-1].copy()
    return off.astype(np.int32), col.astype(np.int32)


@pytest.mark.parametrize("kind", ["first", "all", "decreasing"])
@pytest.mark.parametrize("n", [2, 3, 32, 33, 34, 65, 1025, 300_000])
def test_refused(gpu_lib, n, kind):
    import torch

    t = gpu_lib
    off, col = (torch.from_numpy(a).cuda() for a in _bad(n, kind))
    good = gg.path(n, directed=True)
    fine = (n, torch.from_numpy(good.offsets.view(np.int32)).cuda(), torch.from_numpy(good.cols.view(np.int32)).cuda(), True)
    ctx = t.tkc_create()
    try:
        with pytest.raises(t.TkcError) as e:
            t.tkc_load_csr(ctx, n, off, col, True)
        assert e.value.code == t.TKC_EGRAPH
        with pytest.raises(t.TkcError) as e:
            t.tkc_load_csr_many(ctx, [fine, (n, off, col, True), fine])
        assert e.value.code == t.TKC_EGRAPH and e.value.first_bad == 1
        t.tkc_free_graph(t.tkc_load_csr(ctx, *fine))
    finally:
        t.tkc_destroy(ctx)
