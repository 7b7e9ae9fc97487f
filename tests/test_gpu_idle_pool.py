"""The memory that a context keeps idle is no loss to another context on the
device: a call that finds none gets it.  The rest of the card is held by this
program, as a neighbour's would be."""
import numpy as np
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu
GB = 1 << 30


def test_idle_memory_of_another_context_is_used(gpu_lib):
    import torch

    t = gpu_lib
    n, arcs = 1 << 20, 600_000_000
    off = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    small = gg.path(50)
    torch.cuda.synchronize()
    a, b = t.tkc_create(), t.tkc_create()
    hold = None
    try:
        h = t.tkc_load_csr(b, small.n, small.offsets, small.cols, small.directed)
        t.tkc_topk_closeness(h, 5)  # b has its workspace
        t.tkc_free_graph(h)
        # a takes 2.4 GB of columns (refused: they are not those of the offsets) and keeps them idle
        cols = torch.zeros(arcs, dtype=torch.int32, device="cuda")
        with pytest.raises(t.TkcError) as e:
            t.tkc_load_csr(a, n, off, cols, True)
        assert e.value.code == t.TKC_EGRAPH
        free = torch.cuda.mem_get_info()[0]
        hold = torch.empty(free - GB, dtype=torch.uint8, device="cuda")
        with pytest.raises(t.TkcError) as e:
            t.tkc_load_csr(b, n, off, cols, True)
        assert e.value.code == t.TKC_EGRAPH  # not TKC_ENOMEM: it was copied and checked
        h = t.tkc_load_csr(a, small.n, small.offsets, small.cols, small.directed)
        assert len(t.tkc_topk_closeness(h, 5).ids) == 5
        t.tkc_free_graph(h)
    finally:
        del hold
        torch.cuda.empty_cache()
        t.tkc_destroy(a)
        t.tkc_destroy(b)
