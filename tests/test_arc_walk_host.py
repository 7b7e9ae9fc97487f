"""The warp walk over the arcs of a CSR, its index arithmetic run on the host
(tests/c/arc_walk_host.cpp compiles tkc_arcs.cuh itself): every arc of a valid
CSR is met once with its source, and offsets that no check has seen yet -- a
first offset above 0, decreasing ones, an end below the arcs -- neither keep
the walk from ending nor take a read out of off[0 .. n]."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("walk") / "arc_walk")
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_1704_01077_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "c", "arc_walk_host.cpp"), "-o", exe], check=True, capture_output=True)

    def run(off, a0, a1, check):
        text = "\n".join(str(int(x)) for x in off)
        return subprocess.run([exe, str(len(off) - 1), str(a0), str(a1), "1" if check else "0"], input=text, text=True,
                              timeout=60).returncode

    return run


def _offsets(n, arcs, seed):
    return np.r_[0, np.sort(np.random.default_rng(seed).integers(0, arcs + 1, n - 1)), arcs] if n > 1 else np.array([0, arcs])


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 1023, 1100])
def test_valid_offsets(walk, n):
    off = _offsets(n, 150, n)
    assert walk(off, 0, 150, True) == 0
    assert walk(off, 37, 101, True) == 0


@pytest.mark.parametrize("n", [1, 2, 3, 10, 31, 32, 33, 64, 65, 1023, 1025, 5000])
@pytest.mark.parametrize("kind", ["first", "all", "decreasing", "short", "huge"])
def test_unchecked_offsets_end_within_the_array(walk, n, kind):
    off = _offsets(n, 150, n + 1)
    if kind == "first":
        off[0] = 1
    elif kind == "all":
        off = off + 200
    elif kind == "decreasing":
        off = off[::-1].copy()
    elif kind == "short":
        off = off // 3
    else:
        off = np.full(n + 1, 0xffffffff, np.int64)
    for a0, a1 in ((0, 150), (0, 1), (149, 150)):
        assert walk(off, a0, a1, False) == 0, (a0, a1)
