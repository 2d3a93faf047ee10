// Which form of the first dense stage's split-operand kernel a call takes: plain C++ that a test can compile by itself.
#pragma once

#include <cstdint>

namespace gnnpre {

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
