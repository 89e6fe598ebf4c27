"""The plans of ragged collections kept between calls are bounded in bytes: planning a series of large
collections leaves no more than the stated 32 MB (and the allocator's slack) in use. Host planning only."""
import ctypes

import numpy as np
import pytest


class _MallInfo(ctypes.Structure):
    _fields_ = [(n, ctypes.c_size_t) for n in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks",
                                               "uordblks", "fordblks", "keepcost")]


def test_kept_plans_are_bounded():
    libc = ctypes.CDLL(None)
    if not hasattr(libc, "mallinfo2"):
        pytest.skip("needs glibc's mallinfo2")
    libc.mallinfo2.restype = _MallInfo

    def in_use():
        m = libc.mallinfo2()
        return m.uordblks + m.hblkhd

    from paper_1801_01928_gb300 import build
    path = build.build()
    import paper_1801_01928_gb300 as t3f
    lib, b = t3f.load(path), t3f._binding
    count, group, d = 60000, 20, 6
    dims = np.full(count, d, np.int32)
    modes = np.full(count * d, 2, np.int32)
    ranks = np.tile(np.array([1, 2, 2, 2, 2, 2, 1], np.int32), count)
    gs = np.arange(0, count + 1, group, dtype=np.int32)
    off = np.arange(count, dtype=np.int64) * 40
    ip = ctypes.POINTER(ctypes.c_int32)
    p = lambda a, t=ctypes.c_int32: a.ctypes.data_as(ctypes.POINTER(t))
    before = in_use()
    for v in range(9):
        off += 40  # another collection: the offsets are part of a plan
        desc = b._RDesc(count, p(dims), p(modes), p(ranks), p(off, ctypes.c_int64), ctypes.c_void_p(256), 0)
        assert lib.t3f_gram_groups_workspace_size(ctypes.byref(desc), len(gs) - 1, p(gs), ip()) > 0
    assert in_use() - before < 40 << 20
