"""The workspace does not grow for callers who gain nothing from it: a fan's
tables lie in memory that a call has anyway, so one large set, and many sets
too small for a fan, need no more than they did before sets of a batch had fans
of their own (the figures; a thousandth for the sets' records)."""
import ctypes

import pytest

ch = pytest.importorskip("paper_2303_10581_gb300")


def size(n, sets):
    import os
    if not os.path.exists(ch.library_path()):
        pytest.skip("needs the built library")
    b = ctypes.c_size_t()
    assert ch.load().ch_workspace_size(ctypes.c_int64(n), ctypes.c_int64(sets), ctypes.byref(b)) == 0
    return b.value


@pytest.mark.parametrize("n,sets,most", [
    (1, 1, 1_302_016),
    (10**6, 1, 57_075_968),
    (10**8, 1, 5_273_243_904),
    (10**9, 1, 52_698_760_192),
    (10**7, 1000, 703_565_056),
    (445_000_000, 4096, 25_763_187_200),
    (10**5, 10**5, 10_577_385_728),
    (2 * 10**7, 10**5, 11_765_492_736),
    (10**8, 10**5, 16_541_076_480),
])
def test_size(n, sets, most):
    assert size(n, sets) <= 1.001 * most
