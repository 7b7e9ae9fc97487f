"""Many graphs checked in one launch: each graph has its own part of the grid,
empty graphs none, directed ones none of the symmetry check's.  A planted
fault is reported for the graph that holds it, wherever it sits in the list and
in the graph (first row, last row, a hub row spread over several blocks); a list
without one loads."""
import numpy as np
import pytest

from paper_1704_01077_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(gpu_lib):
    c = gpu_lib.tkc_create()
    yield c
    gpu_lib.tkc_destroy(c)


def _spec(many):
    empty = (0, np.zeros(1, np.uint32), np.zeros(0, np.uint32), False)
    lone = (1, np.zeros(2, np.uint32), np.zeros(0, np.uint32), True)
    gs = [gg.rmat(9, 8, seed=5), gg.barabasi_albert(3000, 4, 6), gg.star(40000), gg.cycle(33, False), gg.path(2, directed=True)]
    spec = [(g.n, g.offsets.astype(np.uint32), g.cols.astype(np.uint32), g.directed) for g in gs]
    out = [empty] + spec[:2] + [empty, lone] + spec[2:] + [empty]
    return out * 40 if many else out


def _fault(kind, g):
    """A copy of g (n >= 3, with arcs) with one fault of the kind."""
    n, off, col, directed = g[0], g[1].copy(), g[2].copy(), g[3]
    if kind == "range":
        col[-1] = n
    elif kind == "self":
        v = int(np.flatnonzero(np.diff(off))[-1])
        col[off[v + 1] - 1] = v
    elif kind == "unsorted":
        v = int(np.argmax(np.diff(off)))
        col[off[v + 1] - 1] = col[off[v + 1] - 2]
    elif kind == "asymmetric":  # drop the last arc
        off[-1] -= 1
        col = col[:-1]
        n, off = n, np.minimum(off, off[-1])
    elif kind == "offsets":
        v = int(np.argmax(np.diff(off)))
        off[v + 1] = off[v] - 1 if off[v] else len(col) + 5
    return n, off, col, directed


@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("kind,which", [("range", 1), ("range", 5), ("self", 2), ("self", 6), ("unsorted", 5),
                                        ("unsorted", 1), ("asymmetric", 2), ("asymmetric", 5), ("asymmetric", 6),
                                        ("offsets", 1), ("offsets", 5), (None, 0)])
def test_faults_are_found_in_their_graph(gpu_lib, ctx, kind, which, many):
    t = gpu_lib
    spec = _spec(many)
    at = which + (len(spec) // 9 - 1) // 2 * 9 if many else which
    if kind is None:
        for h in t.tkc_load_csr_many(ctx, spec):
            t.tkc_free_graph(h)
        return
    spec[at] = _fault(kind, spec[at])
    with pytest.raises(t.TkcError) as e:
        t.tkc_load_csr_many(ctx, spec)
    assert e.value.code == t.TKC_EGRAPH and e.value.first_bad == at
