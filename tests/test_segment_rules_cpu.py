"""The rules of plan construction (csrc/segment_rules.h) and of the first dense stage (csrc/lc_rules.h), compiled for the CPU."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include "segment_rules.h"
#include "lc_rules.h"
extern "C" int rows_asked_ahead(int k_chunks, int64_t tiles, int64_t ctas) { return gnnpre::rows_asked_ahead(k_chunks, tiles, ctas); }
extern "C" int pairs_of_ctas(int64_t hidden, int k_chunks, int resident, int64_t tiles, int num_sms) {
    return gnnpre::pairs_of_ctas(hidden, k_chunks, resident, tiles, num_sms);
}
extern "C" int column_bucket(uint32_t col, int64_t n) { return gnnpre::column_bucket(col, n); }
extern "C" int near_diagonal(uint32_t row, uint32_t col, int64_t n) { return gnnpre::near_diagonal(row, col, n); }
extern "C" int auto_segment_edges(int64_t width, int64_t m, int64_t blocks, int bulk_copy, int beyond, int whole_hops, int num_sms) {
    return gnnpre::auto_segment_edges(width, m, blocks, bulk_copy, beyond, whole_hops, num_sms);
}
extern "C" int64_t count_segments(int64_t m, int64_t blocks, int64_t edges) { return gnnpre::count_segments(m, blocks, edges); }
extern "C" int order_buckets() { return gnnpre::kOrderBuckets; }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fPIC", "-shared", "-I", os.path.join(ROOT, "paper_2207_12000_b200", "csrc"),
                    "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.column_bucket.argtypes = [ctypes.c_uint32, ctypes.c_int64]
    lib.auto_segment_edges.argtypes = [ctypes.c_int64] * 3 + [ctypes.c_int] * 4
    lib.pairs_of_ctas.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    lib.rows_asked_ahead.argtypes = [ctypes.c_int, ctypes.c_int64, ctypes.c_int64]
    lib.count_segments.argtypes, lib.count_segments.restype = [ctypes.c_int64] * 3, ctypes.c_int64
    lib.near_diagonal.argtypes = [ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int64]
    return lib


@pytest.mark.parametrize("n", [1, 2, 1000, 1024, 2449029, 2 ** 31 - 2])
def test_buckets_of_columns_stay_in_range_whatever_the_column(rules, n):
    """Columns are not checked with GNNPRE_FLAG_SKIP_VALIDATION, and the bucket is an index of the plan's tables."""
    B = rules.order_buckets()
    inside = sorted({0, n // 3, n // 2, n - 1})
    for col in inside:
        assert rules.column_bucket(col, n) == col * B // n < B
    for col in (n, n + 1, 2 * n, 2 ** 31 - 1):
        assert rules.column_bucket(min(col, 2 ** 31 - 1), n) == B - 1


def test_near_the_diagonal_is_a_thirty_second_of_all_rows(rules):
    n = 1024 * 100
    for row in (0, 50000, n - 1):
        for apart, near in ((0, 1), (3199, 1), (3400, 0), (60000, 0)):
            for col in (row - apart, row + apart):
                if 0 <= col < n:
                    assert rules.near_diagonal(row, col, n) == near


SMS = 148


@pytest.mark.parametrize("width,m,want", [
    (500, 13264, 16), (500, 10556, 16), (256, 7000, 16), (132, 28000, 16),  # all tiles' segments of 16 edges at once
    (500, 24400, 32), (1433, 13264, 32), (3703, 13264, 32),                 # several waves of them
])
def test_small_graphs_of_several_column_tiles(rules, width, m, want):
    assert rules.auto_segment_edges((width + 3) // 4 * 4, m, 1, 0, 0, 1, SMS) == want
    assert rules.auto_segment_edges((width + 3) // 4 * 4, m, 1, 0, 0, 0, SMS) == 32  # a launch of one block


@pytest.mark.parametrize("m,blocks,edges", [(1, 1, 16), (100, 7, 16), (1000, 32, 31), (1000, 1000, 8), (123457, 256, 40)])
def test_segments_of_all_blocks_are_counted(rules, m, blocks, edges):
    ends = [l * m // blocks for l in range(blocks + 1)]
    assert rules.count_segments(m, blocks, edges) == sum(-(-(hi - lo) // edges) for lo, hi in zip(ends, ends[1:]))


@pytest.mark.parametrize("blocks", [1, 4, 32, 256])
@pytest.mark.parametrize("width,most_edges,most_waves", [(16, 192, 4), (32, 160, 4), (64, 96, 4), (128, 160, 1)])
def test_whole_waves_count_the_blocks(rules, width, most_edges, most_waves, blocks):
    """Segments of a whole hop over few waves: as many waves as the longest segments need, none nearly empty, the shortest such."""
    groups = SMS * 28 * 32 // (width // 4)
    for m in range(50_000, groups * most_edges * most_waves, 7919):
        got = rules.auto_segment_edges(width, m, blocks, 0, 0, 1, SMS)
        waves = -(-rules.count_segments(m, blocks, got) // groups)
        fewest = next((w for w in range(1, most_waves + 1) if rules.count_segments(m, blocks, most_edges) <= groups * w), None)
        if fewest is not None:
            assert got % 8 == 0 and 16 <= got <= most_edges and waves == fewest, m
            assert got == 16 or rules.count_segments(m, blocks, got - 8) > groups * waves or m >= groups * waves * (got - 8), m


@pytest.mark.parametrize("bulk_copy", [0, 1])
def test_long_segments_where_the_order_of_the_sources_is_not_used(rules, bulk_copy):
    """124 M edges in one launch over a matrix beyond the L2: shorter segments where more of them then lie in one row; streamed
    plans (for which the rule is told that nothing is beyond the L2) keep the long ones."""
    for width in (72, 100, 124):
        assert rules.auto_segment_edges(width, 123718280, 1, bulk_copy, 1, 1, SMS) == (1024 if bulk_copy else 512)
        assert rules.auto_segment_edges(width, 123718280, 1, bulk_copy, 0, 0, SMS) == (4096 if bulk_copy else 1024)


@pytest.mark.parametrize("hidden,features,resident,per_sm", [
    (256, 16, 1, None), (192, 64, 1, None), (256, 96, 1, None), (128, 256, 1, None),  # never: few features; one half only
    (192, 65, 1, 24), (192, 96, 1, 24), (256, 97, 1, 12), (192, 97, 1, 8), (192, 160, 1, 8),
    (256, 129, 0, 4), (192, 161, 0, 4), (256, 602, 0, 4),
])
def test_pairs_of_ctas_from_as_many_tiles_as_make_them_faster(rules, hidden, features, resident, per_sm):
    pairs = lambda tiles: rules.pairs_of_ctas(hidden, -(-features // 32), resident, tiles, SMS)
    if per_sm is None:
        assert not pairs(SMS * 10_000)
    else:
        assert pairs(SMS * per_sm) and not pairs(SMS * per_sm - 1)


@pytest.mark.parametrize("k_chunks,per_cta", [(1, 4), (3, 4), (4, 8), (19, 8)])
def test_row_numbers_are_asked_for_ahead_where_a_cta_has_many_tiles(rules, k_chunks, per_cta):
    for ctas in (74, 148):
        assert rules.rows_asked_ahead(k_chunks, per_cta * ctas, ctas) and not rules.rows_asked_ahead(k_chunks, per_cta * ctas - 1, ctas)
