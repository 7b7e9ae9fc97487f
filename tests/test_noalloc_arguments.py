"""tkc_distance_sums_noalloc refuses more sources than vertices before it touches
a device: they cannot be distinct, and a count near 2^32 would take the check's
32-bit positions past their range."""
import ctypes

import pytest


@pytest.mark.parametrize("n,nsrc", [(1, 2), (10, 11), (65536, 65537), (65536, 0xffffffff)])
def test_more_sources_than_vertices(n, nsrc):
    from paper_1704_01077_gb300 import build, tkc

    build.build()
    lib = ctypes.CDLL(build.LIB)
    vp, u32, u64 = ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint64
    fn = lib.tkc_distance_sums_noalloc
    fn.argtypes = [vp, vp, u32, u64, u32, vp, vp, vp, vp]
    some = vp(4096)  # never read
    assert fn(some, some, n, 0, nsrc, some, some, some, None) == tkc.TKC_EINVAL
