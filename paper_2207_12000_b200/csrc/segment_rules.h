// What plan construction decides about segments by arithmetic alone: plain C++ that host and device share, and that a test can
// compile for the CPU.
#pragma once

#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define GNNPRE_HOST_DEVICE __host__ __device__
#else
#define GNNPRE_HOST_DEVICE
#endif

namespace gnnpre {

constexpr int kOrderBuckets = 1024;  // of segments inside one row, by their middle column

// The bucket of a column of n.  A column that nobody has checked (GNNPRE_FLAG_SKIP_VALIDATION) may be any 31-bit number: what
// is out of range goes to the last bucket, so that it is never an index out of a table's range.
GNNPRE_HOST_DEVICE inline int column_bucket(uint32_t col, int64_t n) {
    const int64_t bucket = (int64_t)col * kOrderBuckets / n;
    return bucket < kOrderBuckets ? (int)bucket : kOrderBuckets - 1;
}

// Whether a segment of this row whose middle column this is reads rows numbered like its own, within a thirty-second of all.
GNNPRE_HOST_DEVICE inline bool near_diagonal(uint32_t row, uint32_t col, int64_t n) {
    const int apart = column_bucket(row, n) - column_bucket(col, n);
    return apart <= kOrderBuckets / 32 && apart >= -kOrderBuckets / 32;
}

}  // namespace gnnpre
