"""The bytes of a graph's workspace against the arrays that its queries read
(host arithmetic, no GPU)."""
import ctypes

import pytest

FIXED, REAL = 0, 1


@pytest.fixture(scope="module")
def ubt():
    from paper_2602_14084_gb300 import _build
    _build.build()
    import paper_2602_14084_gb300 as ubt
    return ubt


def size(ubt, n, m, kind=FIXED, flags=0):
    opts = ubt._GraphOpts()
    opts.flags = flags
    sz = ctypes.c_size_t(0)
    assert ubt.lib().ubt_graph_workspace_size(n, m, kind, ctypes.byref(opts), ctypes.byref(sz)) == 0
    return sz.value


@pytest.mark.parametrize("n,m", [(100000, 1000000), (1000000, 9119924), (1 << 12, 1 << 20)])
def test_undirected_rows_without_the_index_hold_no_filter(ubt, n, m):
    # uptr, uadj, ueid, uepos + umir, apair_ptr, apairs, alist, work of the owners, queue of long samples
    arrays = 4 * (n + 1) + 16 * m + 8 * m + 16 * m + 4 * (n + 1) + 8 * m + 4 * n + 8 * n + 8 * 4224
    assert size(ubt, n, m, flags=ubt.UBT_OPT_UNDIRECTED) - size(ubt, n, m) <= arrays + 12 * 256


@pytest.mark.parametrize("n,m", [(100000, 1000000), (1000000, 9119924), (1 << 12, 1 << 20)])
def test_index_is_its_slots_and_a_filter_in_place_of_the_build_arrays(ubt, n, m):
    und = size(ubt, n, m, flags=ubt.UBT_OPT_UNDIRECTED)
    idx = size(ubt, n, m, flags=ubt.UBT_OPT_UNDIRECTED | ubt.UBT_OPT_EDGE_INDEX)
    slots = max(64, 1 << (4 * m - 1).bit_length())
    build_arrays = 33 * n  # at least: what only the build uses
    assert 16 * slots <= idx - und <= 16 * slots + max(0, slots // 4 - build_arrays) + 4096


@pytest.mark.parametrize("n,m", [(100000, 1000000), (1000000, 9119924)])
def test_real_graph_holds_no_row_ids_and_no_kept_counts(ubt, n, m):
    assert size(ubt, n, m, FIXED) - size(ubt, n, m, REAL) >= 8 * m
