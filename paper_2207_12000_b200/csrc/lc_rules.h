// Which form of the first dense stage's split-operand kernel a call takes: plain C++ that a test can compile by itself.
#pragma once

#include <cstdint>

namespace gnnpre {

// Hidden > 128, many tiles: pairs of CTAs that gather each row once (and stream the weight half as often) instead of CTAs
// that take a column half each.  A tile of a pair takes longer, and at few features both are bound by their stores, for
// which the halves' eight stages do better than a pair's four.  us, halves / pairs, three hops, at 6, 9.5, 16, 24, 36, 95 tiles of
// 128 rows x hops per SM:
//   hidden 192, F = 72  41.0 / 47.1, 57.1 / 61.8, 90.3 / 93.9, 136 / 139, 205 / 206, 544 / 525 (64: at 95 408 / 494)
//               F = 96  42.5 / 47.1, 63.4 / 65.6, 101 / 102, 149 / 147, 222 / 217, 583 / 560
//               F = 100 51.2 / 53.2, 75.6 / 74.0, 122 / 114, 179 / 167, 268 / 246, 707 / 632 (160: at 9.5 94.2 / 90.4)
//   hidden 256, F = 64  at 9.5 52.1 / 68.8, 24 119 / 151, 95 453 / 560;  F = 32 at 95 356 / 525
//               F = 96  47.2 / 55.8, 68.0 / 79.0, 108 / 122, 160 / 179, 237 / 262, 620 / 688 (237: 1552 / 1717)
//               F = 100 57.5 / 62.1, 82.2 / 84.2, 135 / 130, 200 / 191, 299 / 282, 780 / 731
//               F = 128 59.4 / 64.6, 86.1 / 89.7, 139 / 141, 206 / 207, 306 / 307, 794 / 798 (237: 2000 / 1968)
// Streamed weight, hidden 256, at 4 and 5: F = 160 53.3 / 47.3, 65.7 / 57.4; F = 300 96.9 / 81.2, 120 / 98.5 (one launch of 157
// tiles: 31 / 35).
// k_chunks: chunks of 32 features; resident: the weight stays in shared memory; tiles: of 128 rows, times the hops of a launch.
inline bool pairs_of_ctas(int64_t hidden, int32_t k_chunks, bool resident, int64_t tiles, int num_sms) {
    if (hidden <= 128 || k_chunks < 3 || (k_chunks == 3 && hidden > 192)) return false;
    const int64_t per_sm = !resident ? 4 : k_chunks == 3 ? 24 : hidden > 192 ? 12 : 8;
    return tiles >= per_sm * num_sms;
}

// Whether a CTA that has its tiles to itself asks for a tile's row numbers while it copies the tile before it.  Otherwise the loads
// stand between two tiles, where the slower issue of MMAs once hid them.  A kernel of a few tiles per CTA pays for the longer
// code instead.  us, three hops, without / with: 1.2 M rows, F = 64, hidden 64 550 / 370, hidden 128 719 / 475; F = 96, hidden 128
// 841 / 640; 200,000 rows, F = 96, hidden 128 148 / 115, F = 128, hidden 64 131 / 119; in column halves, F = 16, hidden 256,
// 600,000 rows 493 / 350; 9.5 tiles per CTA, F = 48, hidden 64 27.4 / 25.1; 4, F = 59 16.4 / 15.8; 3.6, F = 116, hidden 192
// 20.9 / 22.0; 3.3, F = 134, hidden 64 22.8 / 23.4; 6.7, F = 116, hidden 192 31.4 / 32.8; one, F = 116 14.4 / 15.2.
inline bool rows_asked_ahead(int32_t k_chunks, int64_t tiles, int64_t ctas) {
    return tiles >= (k_chunks <= 3 ? 4 : 8) * ctas;
}

}  // namespace gnnpre
